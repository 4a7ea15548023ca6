// C ABI of the EBIC GB300 library: contexts, matrix upload, the pair bitmap and population
// evaluation.  The generation-loop entry points live in evolve.cu.
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <new>
#include <tuple>

#include "internal.h"

namespace {

// Restores the caller's current device when an entry point returns.
struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) {
      cudaGetLastError();
      prev = -1;
    }
    if (prev != dev) cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};

int64_t round_up(int64_t v, int64_t m) { return (v + m - 1) / m * m; }

}  // namespace

// Up to this many freed bytes stay cached in the library pool of a device (beyond it, memory
// goes back to the device at the next synchronisation).
constexpr uint64_t kPoolKeepBytes = 8ull << 30;
constexpr int kPoolDevices = 64;

cudaMemPool_t library_pool() {
  static std::mutex mu;
  static cudaMemPool_t pools[kPoolDevices] = {};
  static bool tried[kPoolDevices] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kPoolDevices) {
    cudaGetLastError();
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(mu);
  if (!tried[dev]) {
    tried[dev] = true;
    int supported = 0;
    if (cudaDeviceGetAttribute(&supported, cudaDevAttrMemoryPoolsSupported, dev) == cudaSuccess &&
        supported) {
      cudaMemPoolProps props = {};
      props.allocType = cudaMemAllocationTypePinned;
      props.handleTypes = cudaMemHandleTypeNone;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      cudaMemPool_t pool = nullptr;
      if (cudaMemPoolCreate(&pool, &props) == cudaSuccess) {
        uint64_t keep = kPoolKeepBytes;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        pools[dev] = pool;
      }
    }
    cudaGetLastError();
  }
  return pools[dev];
}

int resident_blocks(const void *kernel, int threads, size_t smem) {
  static std::mutex mu;
  static std::map<std::tuple<int, const void *, int, size_t>, int> known;
  int dev = 0, nb = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) cudaGetLastError();
  const auto key = std::make_tuple(dev, kernel, threads, smem);
  std::lock_guard<std::mutex> lock(mu);
  const auto it = known.find(key);
  if (it != known.end()) return it->second;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  nb = std::max(nb, 1);
  try {
    known[key] = nb;
  } catch (...) {  // (asked again next time)
  }
  return nb;
}

int ebic_fail(ebic_ctx *ctx, int code, const std::string &msg) {
  if (ctx) ctx->err = msg;
  return code;
}

int ebic_fail_cuda(ebic_ctx *ctx, cudaError_t e, const char *what, const char *file, int line) {
  char buf[512];
  snprintf(buf, sizeof(buf), "%s failed: %s (%s:%d)", what, cudaGetErrorString(e), file, line);
  cudaGetLastError();
  if (ctx) ctx->err = buf;
  return e == cudaErrorMemoryAllocation ? EBIC_ENOMEM : EBIC_ECUDA;
}

bool ebic_is_device_ptr(const void *p) {
  if (!p) return false;
  cudaPointerAttributes attr;
  if (cudaPointerGetAttributes(&attr, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged;
}

// The context's pinned block (see ebic_ctx::pin).  Pinning host memory takes a few hundred
// microseconds, so blocks of closed contexts are kept for the next ones: up to kPinKeep of them (32
// MB), as many as a job server has workers.  (With eight kept, the ninth context open at once and
// those after it took about 100 us longer to make and 130 us longer to close, every time.)
constexpr size_t kPinStatus = 256, kPinIn = 256 << 10, kPinOut = 256 << 10;
static_assert(kPinIn + kPinOut == kPinSpare, "the pinned block's size");
constexpr size_t kPinKeep = 64;
static std::mutex g_pin_mu;
static unsigned char *g_pin_free[kPinKeep];
static size_t g_pin_n = 0;

static unsigned char *take_pin() {
  {
    std::lock_guard<std::mutex> lock(g_pin_mu);
    if (g_pin_n) return g_pin_free[--g_pin_n];
  }
  void *p = nullptr;
  if (cudaHostAlloc(&p, kPinStatus + kPinIn + kPinOut,
                    cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return static_cast<unsigned char *>(p);
}

static void give_pin(unsigned char *p) {  // (no work of the context is left that uses it)
  if (!p) return;
  {
    std::lock_guard<std::mutex> lock(g_pin_mu);
    if (g_pin_n < kPinKeep) {
      g_pin_free[g_pin_n++] = p;
      return;
    }
  }
  cudaFreeHost(p);
}

// Whether p is memory of the device (as ebic_is_device_ptr); EBIC_EINVAL when it is another
// device's.  One query for both.
static int classify_ptr(ebic_ctx *ctx, const void *p, const char *name, bool *is_device) {
  *is_device = false;
  cudaPointerAttributes attr;
  if (cudaPointerGetAttributes(&attr, p) != cudaSuccess) {
    cudaGetLastError();
    return EBIC_OK;
  }
  if (attr.type == cudaMemoryTypeDevice && attr.device != ctx->device)
    return ebic_fail(ctx, EBIC_EINVAL, std::string(name) + " is memory of another device");
  *is_device = attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged;
  return EBIC_OK;
}

// Keeps the word that uploads and population checks report in (ebic_ctx::d_err) zero between calls: a
// call that ends without having read it as zero leaves it cleared.
namespace {
struct ErrWordGuard {
  ebic_ctx *ctx;
  bool clean = false;
  ~ErrWordGuard() {
    if (clean) return;
    if (cudaMemsetAsync(ctx->d_err.p, 0, sizeof(int32_t), ctx->stream) != cudaSuccess)
      cudaGetLastError();
  }
};
}  // namespace

static int check_device_ptr(ebic_ctx *ctx, const void *p, const char *name) {
  cudaPointerAttributes attr;
  if (cudaPointerGetAttributes(&attr, p) != cudaSuccess) {
    cudaGetLastError();
    return EBIC_OK;
  }
  if ((attr.type == cudaMemoryTypeDevice) && attr.device != ctx->device)
    return ebic_fail(ctx, EBIC_EINVAL, std::string(name) + " is memory of another device");
  return EBIC_OK;
}

int ebic_check_eval_params(ebic_ctx *ctx, const ebic_params *p) {
  if (!p) return ebic_fail(ctx, EBIC_EINVAL, "params is NULL");
  if (!(p->ratio_num > 0 && p->ratio_num <= p->ratio_den))
    return ebic_fail(ctx, EBIC_EINVAL, "need 0 < ratio_num <= ratio_den");
  if (p->ratio_den > (1 << 24))
    return ebic_fail(ctx, EBIC_EINVAL, "ratio_den must be <= 2^24");
  if (p->neg_trends != 0 && p->neg_trends != 1)
    return ebic_fail(ctx, EBIC_EINVAL, "neg_trends must be 0 or 1");
  if (p->col_cap < 0 || p->col_cap > 16 || p->min_rows < 0)
    return ebic_fail(ctx, EBIC_EINVAL, "need 0 <= col_cap <= 16 and min_rows >= 0");
  if (p->mode < EBIC_MODE_AUTO || p->mode > EBIC_MODE_STAGED)
    return ebic_fail(ctx, EBIC_EINVAL, "unknown mode");
  if ((p->non_strict != 0 && p->non_strict != 1) || (p->last_kept != 0 && p->last_kept != 1))
    return ebic_fail(ctx, EBIC_EINVAL, "non_strict and last_kept must be 0 or 1");
  if (p->last_kept && p->mode == EBIC_MODE_BITMAP)
    return ebic_fail(ctx, EBIC_EINVAL, "the last-kept pair test has no bitmap form");
  if (p->ipw < 0 || p->ipw > 4 || p->fuse_pairs < -1 || p->fuse_pairs >= EBIC_MAX_LEN)
    return ebic_fail(ctx, EBIC_EINVAL, "ipw must be in [0, 4] and fuse_pairs in [-1, 63]");
  return EBIC_OK;
}

cudaEvent_t prof_event(ebic_ctx *ctx) {
  if (!ctx->prof) return nullptr;
  cudaEvent_t e = nullptr;
  if (!ctx->ev_pool.empty()) {
    e = ctx->ev_pool.back();
    ctx->ev_pool.pop_back();
  } else if (cudaEventCreate(&e) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return e;
}

void prof_push(ebic_ctx *ctx, cudaEvent_t a, cudaEvent_t b, int kernel, double bytes, double ops,
               double units, bool own_a, bool own_b) {
  if (a && b) {
    ctx->pending.push_back(PendingTiming{a, b, kernel, bytes, ops, units, own_a, own_b});
  } else {
    if (a) ctx->ev_pool.push_back(a);
    if (b) ctx->ev_pool.push_back(b);
  }
}

cudaEvent_t prof_begin(ebic_ctx *ctx) {
  if (!ctx->prof) return nullptr;
  cudaEvent_t e = nullptr;
  if (!ctx->ev_pool.empty()) {
    e = ctx->ev_pool.back();
    ctx->ev_pool.pop_back();
  } else if (cudaEventCreate(&e) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  cudaEventRecord(e, ctx->stream);
  return e;
}

void prof_end(ebic_ctx *ctx, cudaEvent_t a, int kernel, double bytes, double ops, double units) {
  if (!a) return;
  cudaEvent_t b = nullptr;
  if (!ctx->ev_pool.empty()) {
    b = ctx->ev_pool.back();
    ctx->ev_pool.pop_back();
  } else if (cudaEventCreate(&b) != cudaSuccess) {
    cudaGetLastError();
    ctx->ev_pool.push_back(a);
    return;
  }
  cudaEventRecord(b, ctx->stream);
  ctx->pending.push_back(PendingTiming{a, b, kernel, bytes, ops, units, true, true});
}

void prof_count(ebic_ctx *ctx, int kernel, int64_t n) {
  if (kernel >= 0 && kernel < EBIC_KERNEL_COUNT && kernel != EBIC_KERNEL_ALL)
    ctx->kst[kernel].launches += n;
  ctx->kst[EBIC_KERNEL_ALL].launches += n;
}

void prof_collect(ebic_ctx *ctx) {
  for (const PendingTiming &t : ctx->pending) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, t.a, t.b) == cudaSuccess) {
      KStats &k = ctx->kst[t.kernel];
      k.timed += 1;
      k.ms += ms;
      k.bytes += t.bytes;
      k.ops += t.ops;
      k.units += t.units;
    } else {
      cudaGetLastError();
    }
    if (t.own_a) ctx->ev_pool.push_back(t.a);
    if (t.own_b) ctx->ev_pool.push_back(t.b);
  }
  ctx->pending.clear();
}

// Validates a CSR population (on the host for host arrays, on the device for device arrays)
// and makes it available on the device.  Host arrays are copied into the context's buffers.
int stage_population(ebic_ctx *ctx, const int32_t *col_idx, const int32_t *offsets, int32_t n_ind,
                     bool want_host_offsets, StagedPop *out) {
  const bool dev_cols = ebic_is_device_ptr(col_idx), dev_off = ebic_is_device_ptr(offsets);
  if (dev_cols != dev_off)
    return ebic_fail(ctx, EBIC_EINVAL, "col_idx and offsets must both be host or both device");
  cudaStream_t s = ctx->stream;
  const int32_t *d_cols = col_idx, *d_off = offsets;
  std::vector<int32_t> &h_off = out->h_off;
  double mean_len = 0.0;
  int64_t total = 0;
  if (!dev_cols) {
    // Host CSR: the offsets are checked here (they size the copy), the columns on the device
    // after the copy, by the kernel that checks device populations (a host loop over every
    // column pair took milliseconds for 8,192 individuals of up to 64 columns).
    for (int32_t i = 0; i < n_ind; ++i) {
      const int64_t L = (int64_t)offsets[i + 1] - offsets[i];
      if (offsets[i] < 0 || L < 2 || L > EBIC_MAX_LEN)
        return ebic_fail(ctx, EBIC_EINVAL, "individual " + std::to_string(i) +
                                               ": length must be in [2, 64]");
    }
    total = (int64_t)offsets[n_ind] - offsets[0];
    mean_len = (double)total / n_ind;
    EBIC_CHECK_CUDA(ctx, ctx->ev_cols.ensure((size_t)(offsets[n_ind]) * 4 + 16, ctx->stream));
    EBIC_CHECK_CUDA(ctx, ctx->ev_off.ensure((size_t)(n_ind + 1) * 4, ctx->stream));
    EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(ctx->ev_cols.p, col_idx, (size_t)offsets[n_ind] * 4,
                                         cudaMemcpyHostToDevice, s));
    EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(ctx->ev_off.p, offsets, (size_t)(n_ind + 1) * 4,
                                         cudaMemcpyHostToDevice, s));
    d_cols = ctx->ev_cols.as<int32_t>();
    d_off = ctx->ev_off.as<int32_t>();
    ErrWordGuard guard{ctx};
    EBIC_CHECK_CUDA(ctx, launch_validate_csr(d_cols, d_off, n_ind, ctx->C,
                                             ctx->d_err.as<int32_t>(), s));
    prof_count(ctx, -1, 1);
    int32_t herr = 0;
    EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(&herr, ctx->d_err.p, 4, cudaMemcpyDeviceToHost, s));
    EBIC_CHECK_CUDA(ctx, cudaStreamSynchronize(s));
    if (herr) return ebic_fail(ctx, EBIC_EINVAL, "invalid chromosome in the population");
    guard.clean = true;
    if (want_host_offsets) h_off.assign(offsets, offsets + n_ind + 1);
  } else {
    // Device CSR: validate on the device before any kernel indexes the matrix with it.
    ErrWordGuard guard{ctx};
    EBIC_CHECK_CUDA(ctx, launch_validate_csr(col_idx, offsets, n_ind, ctx->C,
                                             ctx->d_err.as<int32_t>(), s));
    prof_count(ctx, -1, 1);
    int32_t herr = 0;
    int32_t ends[2] = {0, 0};
    EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(&herr, ctx->d_err.p, 4, cudaMemcpyDeviceToHost, s));
    EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(&ends[0], offsets, 4, cudaMemcpyDeviceToHost, s));
    EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(&ends[1], offsets + n_ind, 4, cudaMemcpyDeviceToHost, s));
    if (want_host_offsets) {
      h_off.resize(n_ind + 1);
      EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(h_off.data(), offsets, (size_t)(n_ind + 1) * 4,
                                           cudaMemcpyDeviceToHost, s));
    }
    EBIC_CHECK_CUDA(ctx, cudaStreamSynchronize(s));
    if (herr) return ebic_fail(ctx, EBIC_EINVAL, "invalid chromosome in the population");
    guard.clean = true;
    total = (int64_t)ends[1] - ends[0];
    mean_len = (double)total / n_ind;
  }

  out->d_cols = d_cols;
  out->d_off = d_off;
  out->total = total;
  out->mean_len = mean_len;
  return EBIC_OK;
}

extern "C" {

int ebic_profile_enable(ebic_ctx *ctx, int32_t on) {
  if (!ctx) return EBIC_EINVAL;
  DeviceGuard g(ctx->device);
  cudaStreamSynchronize(ctx->stream);
  cudaGetLastError();
  prof_collect(ctx);
  if (on) {
    for (KStats &k : ctx->kst) k = KStats();
  }
  ctx->prof = on != 0;
  return EBIC_OK;
}

int ebic_profile_read(ebic_ctx *ctx, int32_t kernel, ebic_kernel_stats *out) {
  if (!ctx || !out || kernel < 0 || kernel >= EBIC_KERNEL_COUNT) return EBIC_EINVAL;
  DeviceGuard g(ctx->device);
  cudaStreamSynchronize(ctx->stream);
  cudaGetLastError();
  prof_collect(ctx);
  const KStats &k = ctx->kst[kernel];
  out->launches = k.launches;
  out->timed_launches = k.timed;
  out->ms = k.ms;
  out->alg_bytes = k.bytes;
  out->alg_ops = k.ops;
  out->units = k.units;
  return EBIC_OK;
}

const char *ebic_version(void) { return "ebic-gb300 0.1 (sm_103a)"; }

void ebic_default_params(ebic_params *p) {
  if (!p) return;
  memset(p, 0, sizeof(*p));
  p->neg_trends = 1;
  p->ratio_num = 85;
  p->ratio_den = 100;
  p->min_rows = 2;
  p->col_cap = 10;
  p->overlap_num = 1;
  p->overlap_den = 2;
  p->n_biclusters = 10;
  p->init_min_len = 2;
  p->init_max_len = 8;
  p->max_len = 20;
  p->pop_size = 800;
  p->elite = 10;
  p->tournament = 4;
  p->max_attempts = 4;
  p->tabu_hit_limit = 800;
  p->seed = 20210710ull;
  p->mode = EBIC_MODE_AUTO;
  p->use_graph = 1;
}

int ebic_create(ebic_ctx **out, int32_t device, void *cuda_stream) {
  if (!out) return EBIC_EINVAL;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess) {
    cudaGetLastError();
    return EBIC_ECUDA;
  }
  if (device < 0 || device >= ndev) return EBIC_EINVAL;
  ebic_ctx *ctx = new (std::nothrow) ebic_ctx();
  if (!ctx) return EBIC_ENOMEM;
  ctx->device = device;
  DeviceGuard g(device);
  int l2 = 0;
  if (cudaDeviceGetAttribute(&ctx->num_sms, cudaDevAttrMultiProcessorCount, device) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, device) != cudaSuccess) {
    cudaGetLastError();
    delete ctx;
    return EBIC_ECUDA;
  }
  ctx->l2_bytes = l2;
  if (cuda_stream) {
    ctx->stream = (cudaStream_t)cuda_stream;
  } else {
    if (cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking) != cudaSuccess) {
      cudaGetLastError();
      delete ctx;
      return EBIC_ECUDA;
    }
    ctx->own_stream = true;
  }
  DevWords *const words[] = {&ctx->d_err, &ctx->d_work, &ctx->d_kerr, &ctx->d_ties};
  // (512 bytes apart, as the pool places separate buffers: packed at 64 bytes, the search's small buffers
  // came to lie elsewhere, and a generation at 20,000 x 500 took 33.4 us in place of 33.0)
  constexpr size_t kWordsApart = 512;
  constexpr size_t kWordsBytes = kWordsApart * sizeof(words) / sizeof(words[0]);
  if (ctx->d_words.ensure(kWordsBytes, ctx->stream) != cudaSuccess ||
      cudaMemsetAsync(ctx->d_words.p, 0, kWordsBytes, ctx->stream) != cudaSuccess ||
      !(ctx->pin = take_pin())) {
    cudaGetLastError();
    ebic_destroy(ctx);
    return EBIC_ENOMEM;
  }
  unsigned char *at = ctx->d_words.as<unsigned char>();
  for (DevWords *w : words) {
    w->p = at;
    at += kWordsApart;
  }
  *out = ctx;
  return EBIC_OK;
}

int ebic_destroy(ebic_ctx *ctx) {
  if (!ctx) return EBIC_OK;
  DeviceGuard g(ctx->device);
  cudaStreamSynchronize(ctx->stream);
  cudaGetLastError();
  gen_state_free(ctx->gen);
  ctx->gen = nullptr;
  DevBuf *bufs[] = {&ctx->keys, &ctx->bitmap, &ctx->stage_x, &ctx->d_words, &ctx->ev_cols,
                    &ctx->ev_off, &ctx->ev_out, &ctx->ev_fit, &ctx->codes, &ctx->planes,
                    &ctx->pair_cnt};
  for (DevBuf *b : bufs) b->release();
  give_pin(ctx->pin);
  prof_collect(ctx);
  for (cudaEvent_t e : ctx->ev_pool) cudaEventDestroy(e);
  for (cudaEvent_t e : ctx->seg_ev) cudaEventDestroy(e);
  if (ctx->copy_stream) cudaStreamDestroy(ctx->copy_stream);
  if (ctx->own_stream) cudaStreamDestroy(ctx->stream);
  delete ctx;
  return EBIC_OK;
}

const char *ebic_last_error(const ebic_ctx *ctx) { return ctx ? ctx->err.c_str() : ""; }

int64_t ebic_bitmap_bytes(int64_t rows, int32_t cols) {
  if (rows < 1 || cols < 1) return 0;
  return (int64_t)cols * cols * (round_up(rows, 128) / 32) * 4;
}

}  // extern "C"

int64_t bitmap_stride(int64_t rows, int32_t cols) {
  const int64_t w = round_up(rows, 128) / 32;
  if (!code_bytes_for(cols)) return w;
  for (int64_t line = 32; line >= 8; line /= 2)
    if (round_up(w, line) - w <= w / 16) return round_up(w, line);
  return w;
}

void ctx_release_buffers(ebic_ctx *ctx) {
  gen_state_free(ctx->gen);
  ctx->gen = nullptr;
  DevBuf *bufs[] = {&ctx->keys, &ctx->bitmap, &ctx->stage_x, &ctx->ev_cols, &ctx->ev_off,
                    &ctx->ev_out, &ctx->ev_fit, &ctx->codes, &ctx->planes, &ctx->pair_cnt};
  for (DevBuf *b : bufs) b->release();
  ctx->have_matrix = false;
  ctx->bitmap_ok = false;
  ctx->pair_cnt_ok = false;
  ctx->codes_ready = false;
  ctx->tuned = false;
  ctx->R = ctx->R_pad = ctx->Wst = ctx->Gst = 0;
  ctx->C = 0;
}

namespace {

// Waits for the uploads of a load and reads their error word.
int read_upload_error(ebic_ctx *ctx, ErrWordGuard *guard) {
  EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(ctx->pin, ctx->d_err.p, sizeof(int32_t),
                                       cudaMemcpyDeviceToHost, ctx->stream));
  EBIC_CHECK_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  int32_t herr = 0;
  memcpy(&herr, ctx->pin, sizeof(herr));
  if (herr) return ebic_fail(ctx, EBIC_ENAN, "matrix holds NaN or Inf");
  guard->clean = true;
  return EBIC_OK;
}

// The context's second stream, for copies beside its kernels, and at least n events between the two.
int ensure_copy_stream(ebic_ctx *ctx, int64_t n) {
  if (!ctx->copy_stream)
    EBIC_CHECK_CUDA(ctx, cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking));
  while ((int64_t)ctx->seg_ev.size() < n) {
    cudaEvent_t e = nullptr;
    EBIC_CHECK_CUDA(ctx, cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    ctx->seg_ev.push_back(e);
  }
  return EBIC_OK;
}

// The segmented load of a row-major host matrix (see ebic_load_matrix): kLoadSegments segments
// of a multiple of 8,192 rows (whole 2,048-row chunks of the planes, whole tiles of every
// kernel), the last one with the padded tail.
constexpr int64_t kLoadSegments = 4;

int load_matrix_segmented(ebic_ctx *ctx, const float *x, int64_t rows, int32_t cols,
                          int64_t R_pad) {
  const bool bitmap = ctx->tuned_mode == EBIC_MODE_BITMAP;
  const int64_t C = cols, Gst = bitmap_stride(rows, cols);
  const int cb = code_bytes_for(cols);
  const int64_t S = code_stride_for(rows, cb);
  cudaStream_t s = ctx->stream;
  EBIC_CHECK_CUDA(ctx, ctx->stage_x.ensure((size_t)rows * C * sizeof(float), s));
  EBIC_CHECK_CUDA(ctx, ctx->codes.ensure((size_t)C * S * cb, s));
  EBIC_CHECK_CUDA(ctx, launch_clear_code_tail(ctx->codes.p, cb, S, R_pad, cols, s));
  if (bitmap) {
    EBIC_CHECK_CUDA(ctx, ctx->planes.ensure((size_t)code_plane_words(cols, Gst) * 4, s));
    EBIC_CHECK_CUDA(ctx, ctx->bitmap.ensure((size_t)(C * C * Gst) * 4, s));
    EBIC_CHECK_CUDA(ctx, prepare_bitmap_eval());
    EBIC_CHECK_CUDA(ctx, ctx->pair_cnt.ensure((size_t)C * C * sizeof(unsigned long long), s));
  }
  const int64_t seg =
      std::max<int64_t>(8192, round_up((R_pad + kLoadSegments - 1) / kLoadSegments, 8192));
  const int64_t n_seg = (R_pad + seg - 1) / seg;
  EBIC_TRY(ensure_copy_stream(ctx, n_seg + 1));
  // the copy stream starts after the context stream's earlier work (which may still read the
  // staging buffer)
  EBIC_CHECK_CUDA(ctx, cudaEventRecord(ctx->seg_ev[n_seg], s));
  EBIC_CHECK_CUDA(ctx, cudaStreamWaitEvent(ctx->copy_stream, ctx->seg_ev[n_seg], 0));
  float *stage = ctx->stage_x.as<float>();
  ErrWordGuard guard{ctx};
  for (int64_t i = 0; i < n_seg; ++i) {
    const int64_t r0 = i * seg, r1 = std::min(R_pad, r0 + seg);
    if (r0 < rows) {
      const int64_t n = std::min(r1, rows) - r0;
      EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(stage + r0 * C, x + r0 * C, (size_t)(n * C) * 4,
                                           cudaMemcpyHostToDevice, ctx->copy_stream));
      EBIC_CHECK_CUDA(ctx, cudaEventRecord(ctx->seg_ev[i], ctx->copy_stream));
      EBIC_CHECK_CUDA(ctx, cudaStreamWaitEvent(s, ctx->seg_ev[i], 0));
    }
    EBIC_CHECK_CUDA(ctx, launch_upload_rows(stage, rows, cols, R_pad, ctx->keys.as<uint32_t>(),
                                            ctx->d_err.as<int32_t>(), r0, r1, s));
    EBIC_CHECK_CUDA(ctx, launch_rank_codes_rows(ctx->keys.as<uint32_t>(), R_pad, cols,
                                                ctx->codes.p, cb, S, ctx->num_sms, r0, r1, s));
    prof_count(ctx, -1, 1);
    prof_count(ctx, EBIC_KERNEL_RANK_CODES, 1);
    if (bitmap) {  // (a segment is a multiple of 2,048 rows: whole chunks of planes)
      EBIC_CHECK_CUDA(ctx, launch_code_planes(ctx->codes.p, cb, S, cols, Gst,
                                              ctx->planes.as<uint32_t>(),
                                              i ? nullptr : ctx->pair_cnt.as<unsigned long long>(),
                                              s, r0 / 2048, r1 < R_pad ? r1 / 2048 : -1));
      prof_count(ctx, -1, 1);
    }
  }
  if (bitmap) {
    EBIC_CHECK_CUDA(ctx, launch_build_bitmap_planes(ctx->planes.as<uint32_t>(), cols, Gst,
                                                    ctx->bitmap.as<uint32_t>(),
                                                    ctx->pair_cnt.as<unsigned long long>(),
                                                    ctx->num_sms, s));
    prof_count(ctx, EBIC_KERNEL_BITMAP_BUILD, 1);
    ctx->tie_state = -1;
  }
  EBIC_TRY(read_upload_error(ctx, &guard));
  ctx->R = rows;
  ctx->C = cols;
  ctx->R_pad = R_pad;
  ctx->Wst = R_pad / 32;
  ctx->Gst = Gst;
  direct_tma_prepare(&ctx->dtma, ctx->keys.as<uint32_t>(), R_pad, cols);
  ctx->code_bytes = cb;
  ctx->code_stride = S;
  ctx->codes_ready = true;
  ctx->bitmap_ok = bitmap;
  ctx->pair_cnt_ok = bitmap;
  ctx->have_matrix = true;
  ctx->err.clear();
  return EBIC_OK;
}

}  // namespace

namespace {

// Pair rows [r0, r1) of the bitmap without their padding, to device memory.
int pack_rows(ebic_ctx *ctx, int64_t r0, int64_t r1, uint32_t *out) {
  EBIC_CHECK_CUDA(ctx, launch_copy_rows(ctx->bitmap.as<uint32_t>() + r0 * ctx->Gst, ctx->Gst,
                                        ctx->Wst, r1 - r0, out, ctx->stream));
  prof_count(ctx, -1, 1);
  return EBIC_OK;
}

// The whole bitmap without its padding, to the host (the caller synchronises the context stream).
// Rows of 2 KB and more by the runtime's strided copy, within 2% of a plain one; it falls behind on
// shorter ones (1,568 bytes: 169 against 192 GB/s, 544 bytes: 85 against 182) and on small bitmaps
// (12.6 MB in 1,264-byte rows: 92 against 79 us).  Those are packed into the loads' staging buffer:
// small ones whole (88 us), others in two halves, a short first piece and then pieces of
// kPackBytes, each copied while the next one is packed (184 and 171 GB/s).
constexpr int64_t kPackWhole = 16 << 20, kPackFirst = 4 << 20, kPackBytes = 64 << 20;

int copy_padded_to_host(ebic_ctx *ctx, uint32_t *out) {
  const int64_t n_rows = (int64_t)ctx->C * ctx->C, row = ctx->Wst * 4;
  const bool whole = n_rows * row <= kPackWhole;
  const int64_t first = whole ? n_rows : kPackFirst / row, per = kPackBytes / row;
  const int64_t n = 1 + (n_rows - first + per - 1) / per;  // pieces
  const int64_t half1 = n > 2 ? per : first;               // (piece 2 is the first one's half again)
  const int64_t staged = half1 + std::min(per, n_rows - first);
  cudaStream_t s = ctx->stream;
  if ((!whole && row >= 2048) ||
      ctx->stage_x.ensure((size_t)(staged * row), s) != cudaSuccess) {
    EBIC_CHECK_CUDA(ctx, cudaMemcpy2DAsync(out, (size_t)row, ctx->bitmap.p, (size_t)ctx->Gst * 4,
                                           (size_t)row, (size_t)n_rows, cudaMemcpyDeviceToHost, s));
    return EBIC_OK;
  }
  if (whole) {
    EBIC_TRY(pack_rows(ctx, 0, n_rows, ctx->stage_x.as<uint32_t>()));
    EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(out, ctx->stage_x.p, (size_t)(n_rows * row),
                                         cudaMemcpyDeviceToHost, s));
    return EBIC_OK;
  }
  EBIC_TRY(ensure_copy_stream(ctx, 4));
  cudaEvent_t *packed = ctx->seg_ev.data(), *copied = packed + 2;
  auto begin = [&](int64_t i) { return i ? std::min(n_rows, first + (i - 1) * per) : 0; };
  for (int64_t i = 0; i <= n; ++i) {
    if (i < n) {  // piece i into its half, once piece i - 2 has left it
      if (i >= 2) EBIC_CHECK_CUDA(ctx, cudaStreamWaitEvent(s, copied[i & 1], 0));
      EBIC_TRY(pack_rows(ctx, begin(i), begin(i + 1),
                         ctx->stage_x.as<uint32_t>() + (i & 1) * half1 * ctx->Wst));
      EBIC_CHECK_CUDA(ctx, cudaEventRecord(packed[i & 1], s));
    }
    if (i > 0) {  // piece i - 1 to the host
      const int64_t r0 = begin(i - 1), r1 = begin(i), h = (i - 1) & 1;
      EBIC_CHECK_CUDA(ctx, cudaStreamWaitEvent(ctx->copy_stream, packed[h], 0));
      EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(out + r0 * ctx->Wst,
                                           ctx->stage_x.as<uint32_t>() + h * half1 * ctx->Wst,
                                           (size_t)((r1 - r0) * row), cudaMemcpyDeviceToHost,
                                           ctx->copy_stream));
      EBIC_CHECK_CUDA(ctx, cudaEventRecord(copied[h], ctx->copy_stream));
    }
  }
  for (int64_t i = n - 2; i < n; ++i)
    EBIC_CHECK_CUDA(ctx, cudaStreamWaitEvent(s, copied[i & 1], 0));
  return EBIC_OK;
}

}  // namespace

extern "C" {

int ebic_load_matrix(ebic_ctx *ctx, const float *x, int64_t rows, int32_t cols, int32_t layout) {
  if (!ctx) return EBIC_EINVAL;
  if (!x) return ebic_fail(ctx, EBIC_EINVAL, "x is NULL");
  if (rows < 1 || cols < 2 || cols > 65535)
    return ebic_fail(ctx, EBIC_EINVAL, "need rows >= 1 and 2 <= cols <= 65535");
  if (layout != EBIC_LAYOUT_ROW_MAJOR && layout != EBIC_LAYOUT_COL_MAJOR)
    return ebic_fail(ctx, EBIC_EINVAL, "unknown layout");
  if (rows > (int64_t(1) << 31) - 128)
    return ebic_fail(ctx, EBIC_EINVAL, "rows must be < 2^31 - 128");
  DeviceGuard g(ctx->device);
  EBIC_TRY(check_device_ptr(ctx, x, "x"));
  // (a matrix of the same shape keeps the autotuner's decisions; sizes that also depend on whether
  // many of its column pairs are tied are set aside where they are used: tuned_sizes_hold)
  if (rows != ctx->R || cols != ctx->C) ctx->tuned = false;
  ctx->have_matrix = false;
  ctx->bitmap_ok = false;
  ctx->pair_cnt_ok = false;
  // A matrix of the same shape keeps the generation loop's buffers and captured graphs (their
  // device addresses and sizes stay valid); the run state is cleared before the next run.
  if (ctx->gen && rows == ctx->R && cols == ctx->C) {
    gen_mark_reset(ctx->gen);
  } else {
    gen_state_free(ctx->gen);
    ctx->gen = nullptr;
  }
  const int64_t R_pad = round_up(rows, 128);
  EBIC_CHECK_CUDA(ctx, ctx->keys.ensure((size_t)cols * R_pad * sizeof(uint32_t), ctx->stream));
  // A host matrix of a shape the autotuner measured, in a form that reads rank codes: the copy
  // goes in segments, and each segment's keys, rank codes and bit planes are built while the
  // next segment is copied; the pair words (bitmap form) follow in one launch over every row.
  if (!ebic_is_device_ptr(x) && layout == EBIC_LAYOUT_ROW_MAJOR && code_bytes_for(cols) &&
      ctx->tuned && ctx->tuned_mode != EBIC_MODE_STAGED && !ctx->prof)
    return load_matrix_segmented(ctx, x, rows, cols, R_pad);
  const float *src = x;
  if (!ebic_is_device_ptr(x)) {
    EBIC_CHECK_CUDA(ctx, ctx->stage_x.ensure((size_t)rows * cols * sizeof(float), ctx->stream));
    EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(ctx->stage_x.p, x, (size_t)rows * cols * sizeof(float),
                                         cudaMemcpyHostToDevice, ctx->stream));
    src = ctx->stage_x.as<float>();
  }
  ErrWordGuard guard{ctx};
  EBIC_CHECK_CUDA(ctx, launch_upload(src, rows, cols, R_pad, layout, ctx->keys.as<uint32_t>(),
                                     ctx->d_err.as<int32_t>(), ctx->stream));
  prof_count(ctx, -1, 1);
  EBIC_TRY(read_upload_error(ctx, &guard));
  ctx->R = rows;
  ctx->C = cols;
  ctx->R_pad = R_pad;
  ctx->Wst = R_pad / 32;
  ctx->Gst = bitmap_stride(rows, cols);
  direct_tma_prepare(&ctx->dtma, ctx->keys.as<uint32_t>(), R_pad, cols);
  // per-row rank codes for the direct form (C <= 1,024), built on the direct form's first use
  ctx->code_bytes = code_bytes_for(cols);
  ctx->code_stride = ctx->code_bytes ? code_stride_for(rows, ctx->code_bytes) : 0;
  ctx->codes_ready = false;
  ctx->have_matrix = true;
  ctx->err.clear();
  return EBIC_OK;
}

int ebic_build_bitmap(ebic_ctx *ctx) {
  if (!ctx) return EBIC_EINVAL;
  if (!ctx->have_matrix) return ebic_fail(ctx, EBIC_ESTATE, "no matrix loaded");
  if (ctx->bitmap_ok) return EBIC_OK;
  DeviceGuard g(ctx->device);
  const size_t bytes = (size_t)ebic_bitmap_bytes(ctx->R, ctx->C);
  EBIC_CHECK_CUDA(ctx, ctx->bitmap.ensure((size_t)ctx->C * ctx->C * ctx->Gst * 4, ctx->stream));
  EBIC_CHECK_CUDA(ctx, prepare_bitmap_eval());
  // With rank codes (C <= 1,024) the words come from the codes' bit planes, else from the keys.
  if (ctx->code_bytes) EBIC_TRY(ensure_codes(ctx));
  // (and the pair counts, C * C words, cleared with the planes and accumulated with the words)
  if (ctx->code_bytes) {
    const size_t nc = (size_t)ctx->C * ctx->C * sizeof(unsigned long long);
    EBIC_CHECK_CUDA(ctx, ctx->pair_cnt.ensure(nc, ctx->stream));
    EBIC_CHECK_CUDA(ctx, ctx->planes.ensure((size_t)code_plane_words(ctx->C, ctx->Gst) * 4,
                                            ctx->stream));
  }
  cudaEvent_t ev = prof_begin(ctx);  // (the planes and the words)
  if (ctx->code_bytes) {
    EBIC_CHECK_CUDA(ctx, launch_code_planes(ctx->codes.p, ctx->code_bytes, ctx->code_stride,
                                            ctx->C, ctx->Gst, ctx->planes.as<uint32_t>(),
                                            ctx->pair_cnt.as<unsigned long long>(),
                                            ctx->stream));
    prof_count(ctx, -1, 1);
    EBIC_CHECK_CUDA(ctx, launch_build_bitmap_planes(ctx->planes.as<uint32_t>(), ctx->C, ctx->Gst,
                                                    ctx->bitmap.as<uint32_t>(),
                                                    ctx->pair_cnt.as<unsigned long long>(),
                                                    ctx->num_sms, ctx->stream));
  } else
    EBIC_CHECK_CUDA(ctx, launch_build_bitmap(ctx->keys.as<uint32_t>(), ctx->R_pad, ctx->C,
                                             ctx->Wst, ctx->bitmap.as<uint32_t>(), ctx->stream));
  prof_end(ctx, ev, EBIC_KERNEL_BITMAP_BUILD, (double)bytes,
           (double)ctx->C * ctx->C * (double)ctx->R, 0.0);
  prof_count(ctx, EBIC_KERNEL_BITMAP_BUILD, 1);
  ctx->tie_state = -1;
  if (ctx->prof) {  // (later work on the stream is ordered after the build anyway)
    EBIC_CHECK_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    prof_collect(ctx);
  }
  ctx->bitmap_ok = true;
  ctx->pair_cnt_ok = ctx->code_bytes != 0;
  return EBIC_OK;
}

int ebic_copy_bitmap(ebic_ctx *ctx, uint32_t *out, int64_t n_words) {
  if (!ctx) return EBIC_EINVAL;
  if (!ctx->bitmap_ok) return ebic_fail(ctx, EBIC_ESTATE, "no bitmap built");
  const int64_t need = ebic_bitmap_bytes(ctx->R, ctx->C) / 4;
  if (!out || n_words < need) return ebic_fail(ctx, EBIC_EINVAL, "output too small");
  DeviceGuard g(ctx->device);
  EBIC_TRY(check_device_ptr(ctx, out, "out"));
  if (ctx->Gst == ctx->Wst) {
    EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(out, ctx->bitmap.p, (size_t)need * 4, cudaMemcpyDefault,
                                         ctx->stream));
  } else if (ebic_is_device_ptr(out)) {  // (the stored rows are padded)
    EBIC_TRY(pack_rows(ctx, 0, (int64_t)ctx->C * ctx->C, out));
  } else {
    EBIC_TRY(copy_padded_to_host(ctx, out));
  }
  EBIC_CHECK_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  return EBIC_OK;
}

int ebic_copy_pair_counts(ebic_ctx *ctx, uint64_t *out, int64_t n) {
  if (!ctx) return EBIC_EINVAL;
  if (!ctx->bitmap_ok || !ctx->pair_cnt_ok)
    return ebic_fail(ctx, EBIC_ESTATE, "no pair counts built (bitmap from rank codes)");
  const int64_t need = (int64_t)ctx->C * ctx->C;
  if (!out || n < need) return ebic_fail(ctx, EBIC_EINVAL, "output too small");
  DeviceGuard g(ctx->device);
  EBIC_TRY(check_device_ptr(ctx, out, "out"));
  EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(out, ctx->pair_cnt.p, (size_t)need * 8, cudaMemcpyDefault,
                                       ctx->stream));
  EBIC_CHECK_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  return EBIC_OK;
}

// The plain form: a launch per individual, which needs the offsets on the host.
static int eval_population_plain(ebic_ctx *ctx, const int32_t *col_idx, const int32_t *offsets,
                                 int32_t n_ind, EvalArgs &a, void *const outs[4]) {
  cudaStream_t s = ctx->stream;
  StagedPop sp;
  EBIC_TRY(stage_population(ctx, col_idx, offsets, n_ind, true, &sp));
  PopView pv{};
  pv.cols = sp.d_cols;
  pv.off = sp.d_off;
  pv.n = n_ind;
  EBIC_CHECK_CUDA(ctx, cudaMemsetAsync(a.rows_pos, 0, (size_t)n_ind * 3 * 4, s));
  cudaEvent_t ev = prof_begin(ctx);
  for (int32_t i = 0; i < n_ind; ++i)
    EBIC_CHECK_CUDA(ctx, launch_eval_plain(a, sp.d_cols + sp.h_off[i],
                                           sp.h_off[i + 1] - sp.h_off[i], i, s));
  prof_end(ctx, ev, EBIC_KERNEL_EVAL, (double)sp.total * (double)ctx->R_pad * 4.0,
           (double)(sp.total - n_ind) * (double)ctx->R * (a.neg ? 2.0 : 1.0),
           (double)n_ind * (double)ctx->R);
  prof_count(ctx, EBIC_KERNEL_EVAL, n_ind);
  EBIC_CHECK_CUDA(ctx, launch_fitness(a, pv, s));
  prof_count(ctx, -1, 1);
  for (int k = 0; k < 3; ++k)
    if (outs[k])
      EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(outs[k], a.rows_pos + (size_t)k * n_ind,
                                           (size_t)n_ind * 4, cudaMemcpyDefault, s));
  if (outs[3])
    EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(outs[3], a.fitness, (size_t)n_ind * 8,
                                         cudaMemcpyDefault, s));
  EBIC_CHECK_CUDA(ctx, cudaStreamSynchronize(s));
  prof_collect(ctx);
  return EBIC_OK;
}

// Whether the device outputs of an evaluation of n individuals can be written as they are: each on its
// type's boundary, and none over another or over the offsets (which the launch that writes them
// reads).  A caller's arena may hold them otherwise.
static bool outputs_apart(void *const outs[4], const bool dev_out[4], size_t n,
                          const int32_t *offsets) {
  const uintptr_t begin[5] = {(uintptr_t)outs[0], (uintptr_t)outs[1], (uintptr_t)outs[2],
                              (uintptr_t)outs[3], (uintptr_t)offsets};
  const size_t bytes[5] = {n * 4, n * 4, n * 4, n * 8, (n + 1) * 4};
  for (int k = 0; k < 4; ++k) {
    if (!outs[k] || !dev_out[k]) continue;
    if (begin[k] % (k == 3 ? 8 : 4)) return false;
    for (int j = k + 1; j < 5; ++j)
      if (begin[j] && (j == 4 || dev_out[j]) && begin[j] < begin[k] + bytes[k] &&
          begin[k] < begin[j] + bytes[j])
        return false;
  }
  return true;
}

// One evaluation is three launches (check and clears, evaluation, fitness and outputs) and one
// synchronisation; the evaluation and the output do nothing when the check failed.  Only where
// AUTO's choice of the form depends on the mean length of a device population, or where the form
// has its operand (bitmap, rank codes) built by this call, is there a second synchronisation, after
// the check.  A small host population goes through the context's pinned
// block, which the first launch reads and the last one writes, instead of through copies.
// (With separate clears, copies and two to three synchronisations, a call took about 90 us more
// than its kernels: 64 individuals on 200 x 20 from host arrays 110 us, now 31; 800 on
// 10,000 x 100 112 and 57 us; 4,096 on 20,000 x 500 by the bitmap 199 and 122 us; 512 on
// 5,001 x 1,500 125 and 62 us.)
int ebic_eval_population(ebic_ctx *ctx, const int32_t *col_idx, const int32_t *offsets,
                         int32_t n_ind, const ebic_params *p, int32_t *rows_pos,
                         int32_t *rows_neg, int32_t *rows_any, uint64_t *fitness) {
  if (!ctx) return EBIC_EINVAL;
  if (!ctx->have_matrix) return ebic_fail(ctx, EBIC_ESTATE, "no matrix loaded");
  EBIC_TRY(ebic_check_eval_params(ctx, p));
  if (n_ind < 0 || n_ind > (1 << 24)) return ebic_fail(ctx, EBIC_EINVAL, "need 0 <= n_ind <= 2^24");
  if (n_ind == 0) return EBIC_OK;
  if (!col_idx || !offsets) return ebic_fail(ctx, EBIC_EINVAL, "col_idx/offsets NULL");
  DeviceGuard g(ctx->device);
  bool dev_cols, dev_off, dev_out[4] = {};
  EBIC_TRY(classify_ptr(ctx, col_idx, "col_idx", &dev_cols));
  EBIC_TRY(classify_ptr(ctx, offsets, "offsets", &dev_off));
  void *outs[4] = {rows_pos, rows_neg, rows_any, fitness};
  for (int k = 0; k < 4; ++k)
    if (outs[k]) EBIC_TRY(classify_ptr(ctx, outs[k], "output", &dev_out[k]));
  if (dev_cols != dev_off)
    return ebic_fail(ctx, EBIC_EINVAL, "col_idx and offsets must both be host or both device");
  cudaStream_t s = ctx->stream;
  const size_t n = (size_t)n_ind;
  EBIC_CHECK_CUDA(ctx, ctx->ev_out.ensure(n * 3 * sizeof(int32_t), s));
  EBIC_CHECK_CUDA(ctx, ctx->ev_fit.ensure(n * sizeof(uint64_t), s));
  int32_t *counts = ctx->ev_out.as<int32_t>(), *sw = ctx->d_work.as<int32_t>();
  EvalArgs a{};
  auto set_args = [&]() {  // (the matrix's fields change with what is built)
    a = eval_args_for(ctx);
    a.neg = p->neg_trends;
    a.non_strict = p->non_strict;
    a.last_kept = p->last_kept;
    a.rnum = p->ratio_num;
    a.rden = p->ratio_den;
    a.min_rows = p->min_rows;
    a.col_cap = p->col_cap;
    a.rows_pos = counts;
    a.rows_neg = counts + n;
    a.rows_any = counts + 2 * n;
    a.fitness = ctx->ev_fit.as<uint64_t>();
    a.work = sw + kSweepWork;
  };
  if (p->mode == EBIC_MODE_PLAIN) {
    set_args();
    return eval_population_plain(ctx, col_idx, offsets, n_ind, a, outs);
  }
  volatile int32_t *status = reinterpret_cast<volatile int32_t *>(ctx->pin);
  int32_t *status_d = reinterpret_cast<int32_t *>(ctx->pin);
  unsigned char *pin_in = ctx->pin + kPinStatus, *pin_out = pin_in + kPinIn;
  const int32_t *src_cols = col_idx, *src_off = offsets;  // what the first launch reads
  const int32_t *d_cols = col_idx, *d_off = offsets;      // what the evaluation reads
  int32_t *copy_cols = nullptr, *copy_off = nullptr;
  int64_t total = 0;
  bool known = false;
  if (!dev_cols) {
    // the offsets are checked here (they size the copy), the columns by the first launch
    for (int32_t i = 0; i < n_ind; ++i) {
      const int64_t L = (int64_t)offsets[i + 1] - offsets[i];
      if (offsets[i] < 0 || L < 2 || L > EBIC_MAX_LEN)
        return ebic_fail(ctx, EBIC_EINVAL, "individual " + std::to_string(i) +
                                               ": length must be in [2, 64]");
    }
    total = (int64_t)offsets[n_ind] - offsets[0];
    known = true;
    const size_t nc = (size_t)offsets[n_ind] * 4, no = (n + 1) * 4;
    EBIC_CHECK_CUDA(ctx, ctx->ev_cols.ensure(nc + 16, s));
    EBIC_CHECK_CUDA(ctx, ctx->ev_off.ensure(no, s));
    d_cols = ctx->ev_cols.as<int32_t>();
    d_off = ctx->ev_off.as<int32_t>();
    if (nc + no <= kPinIn) {
      memcpy(pin_in, offsets, no);
      memcpy(pin_in + no, col_idx, nc);
      src_off = reinterpret_cast<const int32_t *>(pin_in);
      src_cols = reinterpret_cast<const int32_t *>(pin_in + no);
      copy_cols = ctx->ev_cols.as<int32_t>();
      copy_off = ctx->ev_off.as<int32_t>();
    } else {
      EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(ctx->ev_cols.p, col_idx, nc, cudaMemcpyHostToDevice, s));
      EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(ctx->ev_off.p, offsets, no, cudaMemcpyHostToDevice, s));
      src_cols = d_cols;
      src_off = d_off;
    }
  }
  const bool wait_len =
      !known && mode_needs_mean_len(ctx, p->mode, n_ind, 1, p->last_kept);
  auto choose = [&]() {  // (2: any length will do)
    return choose_mode(ctx, p->mode, n_ind, known ? (double)total / n_ind : 2.0, 1, p->last_kept);
  };
  int mode = wait_len ? EBIC_MODE_AUTO : choose();
  // the form's first use on this matrix builds its operand: not for a population that is refused
  const bool builds =
      (mode == EBIC_MODE_BITMAP && !ctx->bitmap_ok) ||
      (direct_form_used(ctx, mode, p) && ctx->code_bytes && !ctx->codes_ready);
  // (the algorithmic work, for the kernel statistics, needs the total too)
  const bool want_ends = wait_len || builds || (!known && ctx->prof);
  status[4] = 0;
  EBIC_CHECK_CUDA(ctx, launch_sweep_prepare(src_cols, src_off, n_ind, ctx->C, counts, sw,
                                            copy_cols, copy_off,
                                            want_ends ? status_d + 2 : nullptr, s));
  prof_count(ctx, -1, 1);
  if (want_ends) {
    EBIC_CHECK_CUDA(ctx, cudaStreamSynchronize(s));
    if (status[4]) {
      EBIC_CHECK_CUDA(ctx, cudaMemsetAsync(sw, 0, 64, s));
      EBIC_CHECK_CUDA(ctx, cudaStreamSynchronize(s));
      return ebic_fail(ctx, EBIC_EINVAL, "invalid chromosome in the population");
    }
    total = (int64_t)status[3] - status[2];
    known = true;
    if (wait_len) mode = choose();
  }
  // from here on a failure leaves the check's word to be cleared
  auto evaluate = [&]() -> int {
    if (mode == EBIC_MODE_BITMAP && !ctx->bitmap_ok) EBIC_TRY(ebic_build_bitmap(ctx));
    if (mode == EBIC_MODE_BITMAP && p->neg_trends && p->ratio_num < p->ratio_den &&
        eval_args_for(ctx).stage_bitmap)
      EBIC_TRY(ensure_tie_state(ctx));
    if (direct_form_used(ctx, mode, p)) EBIC_TRY(ensure_codes(ctx));
    set_args();
    const bool tuned = tuned_sizes_hold(ctx, mode, p);
    a.seg_passes = !tuned                      ? 0
                   : mode == EBIC_MODE_BITMAP ? ctx->seg_bitmap
                   : mode == EBIC_MODE_DIRECT ? ctx->seg_direct
                                              : 0;
    a.ipw = p->ipw > 0 ? p->ipw : (tuned && mode == EBIC_MODE_BITMAP ? ctx->ipw_bitmap : 1);
    PopView pv{};
    pv.cols = d_cols;
    pv.off = d_off;
    pv.n = n_ind;
    pv.stop = sw + kSweepErr;
    const double pairs = (double)(total - n_ind), nd = a.neg ? 2.0 : 1.0;
    cudaEvent_t e0 = prof_begin(ctx);
    EBIC_CHECK_CUDA(ctx, launch_eval_kernel(mode, a, pv, ctx->num_sms, s, true));
    prof_end(ctx, e0, EBIC_KERNEL_EVAL, eval_bytes(ctx, mode, total, n_ind, a.neg),
             pairs * (double)ctx->R * nd, (double)n_ind * (double)ctx->R);
    prof_count(ctx, EBIC_KERNEL_EVAL, 1);
    // device outputs are written in place where the last launch may write them in any order and by
    // whole words (outputs_apart); host outputs come through the pinned block where they fit; the
    // others by copies from the device buffers, once the call is known to be good
    SweepOut o{};
    const bool in_place = outputs_apart(outs, dev_out, n, dev_off ? offsets : nullptr);
    const bool fits = n * 20 <= kPinOut;
    bool copy[4], copies = false;
    for (int k = 0; k < 4; ++k) {
      copy[k] = outs[k] && !(dev_out[k] ? in_place : fits);
      copies |= copy[k];
    }
    for (int k = 0; k < 3; ++k)
      if (outs[k] && !copy[k])
        o.rows[k] = dev_out[k] ? static_cast<int32_t *>(outs[k])
                               : reinterpret_cast<int32_t *>(pin_out + n * 8) + k * n;
    if (fitness)
      o.fitness = copy[3]      ? ctx->ev_fit.as<uint64_t>()
                  : dev_out[3] ? fitness
                               : reinterpret_cast<uint64_t *>(pin_out);
    EBIC_CHECK_CUDA(ctx, launch_sweep_finish(a, pv, sw, o, status_d, s));
    prof_count(ctx, -1, 1);
    EBIC_CHECK_CUDA(ctx, cudaStreamSynchronize(s));
    prof_collect(ctx);
    if (status[0]) return ebic_fail(ctx, EBIC_EINVAL, "invalid chromosome in the population");
    for (int k = 0; k < 3; ++k)
      if (outs[k] && !dev_out[k] && fits)
        memcpy(outs[k], pin_out + n * 8 + (size_t)k * n * 4, n * 4);
    if (fitness && !dev_out[3] && fits) memcpy(fitness, pin_out, n * 8);
    if (copies) {
      for (int k = 0; k < 3; ++k)
        if (copy[k])
          EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(outs[k], counts + (size_t)k * n, n * 4,
                                               cudaMemcpyDefault, s));
      if (copy[3])
        EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(fitness, ctx->ev_fit.p, n * 8, cudaMemcpyDefault, s));
      EBIC_CHECK_CUDA(ctx, cudaStreamSynchronize(s));
    }
    if (status[1]) {
      cudaMemset(ctx->d_kerr.p, 0, 4);
      return ebic_fail(ctx, EBIC_ETIMEOUT, "a bounded device wait expired in the evaluation");
    }
    return EBIC_OK;
  };
  status[0] = status[1] = 0;
  const int st = evaluate();
  if (st != EBIC_OK) {  // (a call that stopped half way may leave the words set)
    cudaMemsetAsync(sw, 0, 64, s);
    cudaStreamSynchronize(s);
    cudaGetLastError();
  }
  return st;
}

}  // extern "C"

// Individuals without ties are looked for where at most 1/8 of the column pairs are tied: an
// individual of np pairs has none with probability (7/8)^np or more, and the look costs every item
// a round trip to the pair counts.
int ensure_tie_state(ebic_ctx *ctx) {
  if (!ctx->bitmap_ok || !ctx->pair_cnt_ok) {
    ctx->tie_state = 0;
    return EBIC_OK;
  }
  if (ctx->tie_state >= 0) return EBIC_OK;
  EBIC_CHECK_CUDA(ctx, launch_count_tied(ctx->pair_cnt.as<unsigned long long>(), ctx->C, ctx->R,
                                         ctx->d_ties.as<int32_t>(), ctx->stream));
  prof_count(ctx, -1, 1);
  volatile int32_t *n = reinterpret_cast<volatile int32_t *>(ctx->pin) + 8;
  EBIC_CHECK_CUDA(ctx, cudaMemcpyAsync(ctx->pin + 32, ctx->d_ties.p, sizeof(int32_t),
                                       cudaMemcpyDeviceToHost, ctx->stream));
  EBIC_CHECK_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  ctx->tie_state = 16 * (int64_t)*n <= (int64_t)ctx->C * (ctx->C - 1);
  return EBIC_OK;
}

int ensure_codes(ebic_ctx *ctx) {
  if (!ctx->code_bytes || ctx->codes_ready) return EBIC_OK;
  const int64_t S = ctx->code_stride, C = ctx->C;
  EBIC_CHECK_CUDA(ctx, ctx->codes.ensure((size_t)C * S * ctx->code_bytes, ctx->stream));
  cudaEvent_t ev = prof_begin(ctx);
  EBIC_CHECK_CUDA(ctx, launch_rank_codes(ctx->keys.as<uint32_t>(), ctx->R_pad, ctx->C,
                                         ctx->codes.p, ctx->code_bytes, S, ctx->num_sms,
                                         ctx->stream));
  // algorithmic bytes: keys read, codes written
  prof_end(ctx, ev, EBIC_KERNEL_RANK_CODES,
           (double)C * ctx->R_pad * 4.0 + (double)C * S * ctx->code_bytes,
           (double)C * ctx->R_pad, (double)ctx->R_pad);
  prof_count(ctx, EBIC_KERNEL_RANK_CODES, 1);
  if (ctx->prof) {  // (later work on the stream is ordered after the build anyway)
    EBIC_CHECK_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    prof_collect(ctx);
  }
  ctx->codes_ready = true;
  return EBIC_OK;
}

int direct_form_used(const ebic_ctx *ctx, int mode, const ebic_params *p) {
  if (mode == EBIC_MODE_DIRECT) return 1;
  return mode == EBIC_MODE_STAGED && (!ctx->dtma.ok || p->non_strict || p->last_kept);
}


// Evaluation-kernel choice for EBIC_MODE_AUTO: a cost model in row-words, refined by the
// autotuner when it has measured this matrix.  The bitmap costs a one-off build of C^2 * Wst
// words and then (L-1) * Wst words per individual and direction; the direct form gathers
// L * R_pad keys per individual.
EvalArgs eval_args_for(const ebic_ctx *ctx) {
  EvalArgs a{};
  a.keys = ctx->keys.as<uint32_t>();
  a.bitmap = ctx->bitmap_ok ? ctx->bitmap.as<uint32_t>() : nullptr;
  a.pair_cnt = ctx->bitmap_ok && ctx->pair_cnt_ok ? ctx->pair_cnt.as<unsigned long long>() : nullptr;
  a.tie_free = a.pair_cnt && ctx->tie_state == 1;
  a.R = ctx->R;
  a.R_pad = ctx->R_pad;
  a.Wst = ctx->Gst;
  a.C = ctx->C;
  a.err = ctx->d_kerr.as<int32_t>();
  a.dtma = ctx->dtma.ok ? &ctx->dtma : nullptr;
  a.codes = ctx->codes_ready ? ctx->codes.as<uint8_t>() : nullptr;
  a.code_bytes = ctx->codes_ready ? ctx->code_bytes : 0;
  a.S = ctx->codes_ready ? ctx->code_stride : 0;
  a.stage_bitmap = ctx->bitmap_ok && bitmap_stored_bytes(ctx->R, ctx->C) > ctx->l2_bytes;
  a.ipw = 1;
  return a;
}

int64_t eval_passes(const ebic_ctx *ctx, int mode) {
  if (mode == EBIC_MODE_BITMAP) return (ctx->Gst + 127) / 128;
  if (ctx->codes_ready) return ctx->code_stride / code_rows_per_pass(ctx->code_bytes);
  return ctx->R_pad / 128;
}

double eval_bytes(const ebic_ctx *ctx, int mode, int64_t total_len, int64_t n_ind, int neg) {
  // algorithmic bytes of one sweep: the pair words (bitmap), else one code or key per row and
  // chromosome column (the staged form reads each tile of keys once per group of individuals;
  // its algorithmic gathers are counted like the key form's)
  if (mode == EBIC_MODE_BITMAP)
    return (double)(total_len - n_ind) * (double)ctx->Wst * 4.0 * (neg ? 2.0 : 1.0);
  if (mode == EBIC_MODE_DIRECT && ctx->codes_ready)
    return (double)total_len * (double)ctx->code_stride * ctx->code_bytes;
  return (double)total_len * (double)ctx->R_pad * 4.0;
}

int choose_mode(const ebic_ctx *ctx, int requested, int64_t n_ind, double mean_len,
                int expected_sweeps, int last_kept) {
  if (requested != EBIC_MODE_AUTO) return requested;
  if (last_kept) {  // no bitmap form
    return ctx->tuned && ctx->tuned_mode != EBIC_MODE_BITMAP ? ctx->tuned_mode : EBIC_MODE_DIRECT;
  }
  if (ctx->tuned) return ctx->tuned_mode;
  if (ctx->bitmap_ok) return EBIC_MODE_BITMAP;
  if (!cost_model_prefers_bitmap((double)ctx->R_pad, (double)ctx->C, ctx->code_bytes,
                                 (double)n_ind, mean_len, (double)expected_sweeps))
    return EBIC_MODE_DIRECT;
  // (the query of the free memory is slow: only where a bitmap is wanted)
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
    cudaGetLastError();
    free_b = 0;
  }
  const double need = (double)bitmap_build_bytes(ctx->R, ctx->C);
  return need > 0.5 * (double)free_b ? EBIC_MODE_DIRECT : EBIC_MODE_BITMAP;
}

bool mode_needs_mean_len(const ebic_ctx *ctx, int requested, int64_t n_ind, int expected_sweeps,
                         int last_kept) {
  if (requested != EBIC_MODE_AUTO || last_kept || ctx->tuned || ctx->bitmap_ok) return false;
  auto prefers = [&](double mean_len) {
    return cost_model_prefers_bitmap((double)ctx->R_pad, (double)ctx->C, ctx->code_bytes,
                                     (double)n_ind, mean_len, (double)expected_sweeps);
  };
  return prefers(2.0) != prefers((double)std::min<int32_t>(EBIC_MAX_LEN, ctx->C));
}
