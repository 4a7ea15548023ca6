// Population evaluation without any memory allocation (ebic_eval_population_noalloc).
//
// Some callers cannot let a library call cudaMalloc or cudaFree.  Examples: a serving process
// whose framework has already reserved the GPU's memory in its own pool, where a further
// allocation fails or fragments the pool; and latency-critical callers, for whom cudaFree's
// device-wide synchronisation and the allocator's unbounded latency are not acceptable.  This
// entry point takes every input and output from the caller, and keeps its scratch (per-individual
// count accumulators and an error word) in one file-scope `static __device__` array of fixed size,
// which every GPU that loads the library holds until the process exits.
//
// A call is three launches and one synchronisation: k_na_prepare checks the matrix and the
// population and clears the accumulators, k_na_eval counts, k_na_finish writes the outputs.  The
// later two find the error word set and do nothing when the check failed; the host reads it at
// the end.  (With the result of the check read back before the evaluation, clears as separate
// operations, and the evaluation one row per lane from a queue of items on one counter, a call
// took 329 us at 10,000 x 100, 800 individuals: 214 us of it in the evaluation.)
//
// Host code cannot name that array's device address directly: in host code its name stands for
// a host-side shadow.  The address is therefore fetched once per device with
// cudaGetSymbolAddress (with that device current) and handed to the kernels.
//
// CUDA loads modules lazily by default, so this file's module (the array and the kernels' code)
// is placed in device memory only when first used on a device.  The first call on each device
// therefore does that set-up explicitly: it resolves the array's address and queries every
// kernel's attributes, which loads all of them.  Later calls on that device load nothing.
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <mutex>

#include "csr.cuh"
#include "internal.h"
#include "trend.cuh"

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kNaWarps = 8;
constexpr int kNaThreads = kNaWarps * 32;
constexpr int kNaEvalWarps = 32;  // of the evaluation: one block per SM
constexpr int kNaEvalThreads = kNaEvalWarps * 32;
constexpr int kMaxDevices = 64;

struct NoAllocScratch {
  int32_t counts[3 * EBIC_NOALLOC_MAX_IND];  // rows_pos | rows_neg | rows_any accumulators
  int32_t reserved;
  int32_t err;  // 1: non-finite matrix value, 2: bad chromosome; 0 between calls
};

static __device__ __align__(256) NoAllocScratch g_noalloc_scratch;

std::mutex g_setup_mu;
NoAllocScratch *g_scratch_addr[kMaxDevices] = {};

__device__ __forceinline__ int threshold(int L, int num, int den) {
  return (num * (L - 1) + den - 1) / den;
}

// Waits for the preceding kernel of a programmatic launch (no-op otherwise).
__device__ __forceinline__ void wait_prior_grid() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ bool not_finite(uint32_t u) { return (u & 0x7F800000u) == 0x7F800000u; }

// Checks the population (a warp per individual) and the matrix for NaN/Inf (16-byte loads from
// the first 16-byte boundary on, any alignment of x), and clears the accumulators.
// Bound: HBM (one read of x).
__global__ void __launch_bounds__(kNaThreads) k_na_prepare(const float *__restrict__ x,
                                                           int64_t total,
                                                           const int32_t *__restrict__ cols,
                                                           const int32_t *__restrict__ off,
                                                           int32_t n, int32_t C,
                                                           NoAllocScratch *sc) {
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  for (int64_t q = tid; q < 3 * (int64_t)n; q += stride) sc->counts[q] = 0;
  bool bad = false;
  for (int64_t i = tid >> 5; i < n; i += stride >> 5) {  // (whole warps)
    int c0, c1;
    bad |= csr_bad(cols, off[i], off[i + 1], C, lane, &c0, &c1);
  }
  const uint32_t *u = reinterpret_cast<const uint32_t *>(x);
  int64_t head = (int64_t)((16 - (reinterpret_cast<uintptr_t>(x) & 15)) & 15) / 4;
  if (head > total) head = total;
  const int64_t vecs = (total - head) / 4;
  const uint4 *v = reinterpret_cast<const uint4 *>(u + head);
  bool bad_x = false;
#pragma unroll 4
  for (int64_t q = tid; q < vecs; q += stride) {
    const uint4 w = __ldg(v + q);
    bad_x |= not_finite(w.x) || not_finite(w.y) || not_finite(w.z) || not_finite(w.w);
  }
  // the up to three values on either side of the 16-byte pieces
  const int64_t tail0 = head + 4 * vecs;
  if (tid < head) bad_x |= not_finite(__ldg(u + tid));
  if (tid < total - tail0) bad_x |= not_finite(__ldg(u + tail0 + tid));
  const unsigned e = (__any_sync(kFull, bad_x) ? 1u : 0u) | (__any_sync(kFull, bad) ? 2u : 0u);
  if (e && lane == 0) atomicOr(&sc->err, (int)e);
}

// Direct float32 comparisons (-0 equals +0; no FTZ in this file's compilation).  An item is an
// individual and a segment of 128-row passes, segment-major.  A block (one per SM, up to every warp
// the SM holds) owns a run of consecutive items, taken by its warps from a counter in shared
// memory: its individuals read the same rows' pieces of the columns, largely from L1, and uneven
// lengths even out within the block.  A lane counts four rows of a pass: consecutive ones by one
// 16-byte load per column where every column starts on a 16-byte boundary (VEC: x aligned, R a
// multiple of 4), else rows 32 apart by four 4-byte loads (coalesced whatever the alignment).
// NS / LK are the pair-test variants of trend.cuh.
// Bound: instruction issue (83% of cycles at 10,000 x 100, the ALU pipe 75%; the values come from L1,
// 93% hits): comparisons and additions per row, pair and direction.  Whole calls: 108 us
// at 10,000 x 100, 800 individuals of 2-20 columns (116 with the items dealt to all warps of the
// grid in turn, 329 with a row per lane and 32-row items from one global counter), 0.90 ms at
// 30,000 x 300, 4,000 individuals of 2-40 (1.05 dealt in turn).
template <bool NEG, bool NS, bool LK, bool VEC>
__global__ void __launch_bounds__(kNaEvalThreads, 1)
    k_na_eval(const float *__restrict__ x, int64_t R, const int32_t *__restrict__ cols,
              const int32_t *__restrict__ off, int32_t n, int32_t n_seg, int32_t seg_passes,
              int32_t rnum, int32_t rden, NoAllocScratch *sc) {
  __shared__ int64_t s_base[kNaEvalWarps][EBIC_MAX_LEN];
  __shared__ unsigned long long s_next;  // items of the block taken so far
  wait_prior_grid();
  if (sc->err) return;  // (a bad population is never indexed with)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_next = blockDim.x >> 5;
  __syncthreads();
  const int64_t passes_total = (R + 127) / 128;
  const int64_t n_items = (int64_t)n * n_seg;
  const int64_t q0 = n_items * blockIdx.x / gridDim.x;
  const int64_t mine = n_items * (blockIdx.x + 1) / gridDim.x - q0;
  for (int64_t d = warp; d < mine;) {
    const int64_t q = q0 + d;
    const int seg = (int)(q / n), i = (int)(q - (int64_t)seg * n);
    const int st = off[i], L = off[i + 1] - st;
    __syncwarp();
    for (int k = lane; k < L; k += 32) s_base[warp][k] = (int64_t)cols[st + k] * R;
    __syncwarp();
    const int t = threshold(L, rnum, rden);
    const int64_t p0 = (int64_t)seg * seg_passes;
    const int64_t p1 = min(p0 + seg_passes, passes_total);
    int cp = 0, cn = 0, ca = 0;
    for (int64_t pass = p0; pass < p1; ++pass) {
      const int64_t r0 = pass * 128 + (VEC ? 4 * lane : lane);
      const int step = VEC ? 1 : 32;  // the lane's rows: r0 + j * step
      // column k's four values (0 past the last row)
      auto load = [&](int k, float (&v)[4]) {
        const float *p = x + s_base[warp][k] + r0;
        if (VEC) {
          const float4 f = r0 < R ? __ldg(reinterpret_cast<const float4 *>(p))
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
          v[0] = f.x;
          v[1] = f.y;
          v[2] = f.z;
          v[3] = f.w;
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] = r0 + 32 * j < R ? __ldg(p + 32 * j) : 0.f;
        }
      };
      RowTrend<float, NEG, NS, LK> tr[4];
      float v[4];
      load(0, v);
#pragma unroll
      for (int j = 0; j < 4; ++j) tr[j].start(v[j]);
#pragma unroll 4
      for (int k = 1; k < L; ++k) {
        load(k, v);
#pragma unroll
        for (int j = 0; j < 4; ++j) tr[j].step(v[j]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool valid = r0 + j * step < R;
        const bool po = valid && tr[j].inc >= t, ne = valid && NEG && tr[j].dec >= t;
        cp += po;
        cn += ne;
        ca += po || ne;
      }
    }
    cp = __reduce_add_sync(kFull, cp);
    cn = __reduce_add_sync(kFull, cn);
    ca = __reduce_add_sync(kFull, ca);
    if (lane == 0) {
      if (cp) atomicAdd(&sc->counts[i], cp);
      if (cn) atomicAdd(&sc->counts[n + i], cn);
      if (ca) atomicAdd(&sc->counts[2 * n + i], ca);
    }
    unsigned long long nx = 0;
    if (lane == 0) nx = atomicAdd(&s_next, 1ull);
    d = (int64_t)__shfl_sync(kFull, nx, 0);
  }
}

__global__ void k_na_finish(const int32_t *__restrict__ off, int32_t n, int32_t min_rows,
                            int32_t col_cap, const NoAllocScratch *sc, int32_t *rows_pos,
                            int32_t *rows_neg, int32_t *rows_any, uint64_t *fitness) {
  wait_prior_grid();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || sc->err) return;
  const int rp = sc->counts[i], rn = sc->counts[n + i], ra = sc->counts[2 * n + i];
  if (rows_pos) rows_pos[i] = rp;
  if (rows_neg) rows_neg[i] = rn;
  if (rows_any) rows_any[i] = ra;
  if (fitness) {
    const int L = off[i + 1] - off[i];
    const int sh = L < col_cap ? L : col_cap;
    fitness[i] = ra < min_rows ? 0ull : ((uint64_t)ra << sh);
  }
}

using NaKernel = void (*)(const float *, int64_t, const int32_t *, const int32_t *, int32_t,
                          int32_t, int32_t, int32_t, int32_t, NoAllocScratch *);
// Indexed by neg_trends * 8 + non_strict * 4 + last_kept * 2 + aligned.
#define EBIC_NA(NEG, NS) \
  k_na_eval<NEG, NS, false, false>, k_na_eval<NEG, NS, false, true>, \
      k_na_eval<NEG, NS, true, false>, k_na_eval<NEG, NS, true, true>
const NaKernel kNaEval[16] = {EBIC_NA(false, false), EBIC_NA(false, true), EBIC_NA(true, false),
                              EBIC_NA(true, true)};
#undef EBIC_NA

// Launches `kern` so that it may be scheduled while the previous kernel of the stream drains (it
// waits for that kernel's results before it reads them).
template <class... Args>
cudaError_t launch_next(void (*kern)(Args...), unsigned grid, unsigned block, cudaStream_t s,
                        Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

int g_num_sms[kMaxDevices] = {};  // set with the scratch address

// Set-up for `device`, done once: with the device current, fetch the device address of the
// scratch array and query every kernel of this file, so that the module (array and code) is in
// device memory before the call returns.  Returns the cached address on later calls.
cudaError_t scratch_for_device(int device, NoAllocScratch **out) {
  std::lock_guard<std::mutex> lock(g_setup_mu);
  if (!g_scratch_addr[device]) {
    int prev = -1;
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    cudaError_t e = cudaSetDevice(device);
    if (e != cudaSuccess) return e;
    void *ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_na_prepare);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_na_finish);
    for (int k = 0; k < 16 && e == cudaSuccess; ++k) e = cudaFuncGetAttributes(&fa, kNaEval[k]);
    if (e == cudaSuccess)
      e = cudaDeviceGetAttribute(&g_num_sms[device], cudaDevAttrMultiProcessorCount, device);
    if (prev >= 0 && prev != device) cudaSetDevice(prev);
    if (e != cudaSuccess) return e;
    g_scratch_addr[device] = static_cast<NoAllocScratch *>(ptr);
  }
  *out = g_scratch_addr[device];
  return cudaSuccess;
}

int fail(char *msg, int32_t msg_len, int code, const char *text) {
  if (msg && msg_len > 0) snprintf(msg, (size_t)msg_len, "%s", text);
  return code;
}

bool on_device(const void *p, int device) {
  cudaPointerAttributes a;
  if (!p || cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) &&
         (a.type == cudaMemoryTypeManaged || a.device == device);
}

}  // namespace

extern "C" int ebic_eval_population_noalloc(const float *x, int64_t rows, int32_t cols,
                                            const int32_t *col_idx, const int32_t *offsets,
                                            int32_t n_ind, const ebic_params *p,
                                            int32_t *rows_pos, int32_t *rows_neg,
                                            int32_t *rows_any, uint64_t *fitness,
                                            int32_t device, void *cuda_stream, char *msg,
                                            int32_t msg_len) {
  if (msg && msg_len > 0) msg[0] = '\0';
  if (!p) return fail(msg, msg_len, EBIC_EINVAL, "params is NULL");
  if (!(p->ratio_num > 0 && p->ratio_num <= p->ratio_den) || p->ratio_den > (1 << 24))
    return fail(msg, msg_len, EBIC_EINVAL, "need 0 < ratio_num <= ratio_den <= 2^24");
  if ((p->neg_trends != 0 && p->neg_trends != 1) || p->col_cap < 0 || p->col_cap > 16 ||
      p->min_rows < 0)
    return fail(msg, msg_len, EBIC_EINVAL, "bad neg_trends, col_cap or min_rows");
  if ((p->non_strict != 0 && p->non_strict != 1) || (p->last_kept != 0 && p->last_kept != 1))
    return fail(msg, msg_len, EBIC_EINVAL, "non_strict and last_kept must be 0 or 1");
  if (rows < 1 || rows > (int64_t(1) << 31) - 32 || cols < 2 || cols > 65535)
    return fail(msg, msg_len, EBIC_EINVAL, "need 1 <= rows < 2^31 - 32 and 2 <= cols <= 65535");
  if (n_ind < 0 || n_ind > EBIC_NOALLOC_MAX_IND)
    return fail(msg, msg_len, EBIC_EINVAL,
                "n_ind is beyond EBIC_NOALLOC_MAX_IND (65536), the size of the static scratch");
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess) {
    cudaGetLastError();
    return fail(msg, msg_len, EBIC_ECUDA, "cudaGetDeviceCount failed");
  }
  if (device < 0 || device >= ndev || device >= kMaxDevices)
    return fail(msg, msg_len, EBIC_EINVAL, "bad device");
  if (n_ind == 0) return EBIC_OK;
  if (!on_device(x, device) || !on_device(col_idx, device) || !on_device(offsets, device))
    return fail(msg, msg_len, EBIC_EINVAL,
                "x, col_idx and offsets must be device memory of `device`");
  void *outs[4] = {rows_pos, rows_neg, rows_any, fitness};
  for (void *o : outs)
    if (o && !on_device(o, device))
      return fail(msg, msg_len, EBIC_EINVAL, "outputs must be device memory of `device`");

  NoAllocScratch *sc = nullptr;
  cudaError_t e = scratch_for_device(device, &sc);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(msg, msg_len, EBIC_ECUDA,
                "set-up failed: the scratch array's address or the kernels could not be loaded");
  }
  int prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess) {
    cudaGetLastError();
    prev = -1;
  }
  if (prev != device && (e = cudaSetDevice(device)) != cudaSuccess) {
    cudaGetLastError();
    return fail(msg, msg_len, EBIC_ECUDA, "cudaSetDevice failed");
  }
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  int status = EBIC_OK;
  do {
    const int64_t num_sms = g_num_sms[device], total = rows * (int64_t)cols;
    const int64_t pre = std::max((total / 16 + kNaThreads - 1) / kNaThreads,
                                 (int64_t)(n_ind + kNaWarps - 1) / kNaWarps);
    k_na_prepare<<<(unsigned)std::min<int64_t>(pre, 8 * num_sms), kNaThreads, 0, s>>>(
        x, total, col_idx, offsets, n_ind, cols, sc);
    if ((e = cudaGetLastError()) != cudaSuccess) break;
    // Segments: about six items per warp, so that the uneven lengths even out.  10,000 x 100 and
    // 30,000 x 300, as above: 108 us and 0.90 ms; with three items 109 and 0.98, with ten 116 and
    // 0.85; segments of one pass 113 us and 0.91 ms.
    const int64_t passes_total = (rows + 127) / 128;
    int64_t seg = ((int64_t)n_ind * passes_total) / (6 * num_sms * kNaEvalWarps);
    if (seg < 1) seg = 1;
    if (seg > passes_total) seg = passes_total;
    const int64_t n_seg = (passes_total + seg - 1) / seg;
    const int64_t items = (int64_t)n_ind * n_seg, grid = std::min<int64_t>(items, num_sms);
    const int64_t warps = std::min<int64_t>((items + grid - 1) / grid, kNaEvalWarps);
    const int aligned = rows % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
    const NaKernel kern = kNaEval[(p->neg_trends ? 8 : 0) + (p->non_strict ? 4 : 0) +
                                  (p->last_kept ? 2 : 0) + aligned];
    if ((e = launch_next(kern, (unsigned)grid, (unsigned)warps * 32u, s, x, rows, col_idx, offsets, n_ind,
                         (int32_t)n_seg, (int32_t)seg, p->ratio_num, p->ratio_den, sc)) !=
        cudaSuccess)
      break;
    if ((e = launch_next(k_na_finish, (unsigned)((n_ind + 255) / 256), 256u, s, offsets, n_ind,
                         p->min_rows, p->col_cap, (const NoAllocScratch *)sc, rows_pos, rows_neg,
                         rows_any, fitness)) != cudaSuccess)
      break;
    int32_t herr = 0;
    if ((e = cudaMemcpyAsync(&herr, &sc->err, sizeof(herr), cudaMemcpyDeviceToHost, s)) !=
        cudaSuccess)
      break;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) break;
    if (herr) {  // (the word is 0 between calls)
      if ((e = cudaMemsetAsync(&sc->err, 0, sizeof(herr), s)) != cudaSuccess) break;
      if ((e = cudaStreamSynchronize(s)) != cudaSuccess) break;
      status = (herr & 1) ? fail(msg, msg_len, EBIC_ENAN, "matrix holds NaN or Inf")
                          : fail(msg, msg_len, EBIC_EINVAL, "invalid chromosome in the population");
    }
  } while (false);
  if (prev >= 0 && prev != device) cudaSetDevice(prev);
  if (e != cudaSuccess) {
    cudaGetLastError();
    cudaMemsetAsync(&sc->err, 0, sizeof(int32_t), s);  // (whatever stopped the call)
    cudaGetLastError();
    char buf[256];
    snprintf(buf, sizeof(buf), "CUDA error: %s", cudaGetErrorString(e));
    return fail(msg, msg_len, EBIC_ECUDA, buf);
  }
  return status;
}
