// Matrix upload (order keys, column-major) and the column-pair comparison bitmap.
//
// Order key: the float32 bit pattern u, with -0 mapped to +0, becomes
//   k(u) = u ^ 0xFFFFFFFF for negative values, u | 0x80000000 otherwise,
// an increasing map of the finite floats onto uint32, so `k(a) > k(b)` is exactly `a > b`
// (ties, including -0 against +0, compare equal) whatever the FTZ/DAZ mode of the arithmetic.
// The trend definition the keys serve is Sec. 2.3 ("EBIC" paragraph) of the EBIC.jl paper.
#include <algorithm>

#include "internal.h"

namespace {

constexpr uint32_t kSign = 0x80000000u;
constexpr uint32_t kExpMask = 0x7F800000u;

__device__ __forceinline__ uint32_t order_key(uint32_t u) {
  if (u == kSign) u = 0u;
  return (u & kSign) ? ~u : (u | kSign);
}

__device__ __forceinline__ bool not_finite(uint32_t u) { return (u & kExpMask) == kExpMask; }

// Row-major x[R][C] -> keys[C][R_pad] through a 32x32 shared-memory tile (coalesced on both
// sides).  Rows in [R, R_pad) get key 0, which never compares greater than anything.
// (rows [r_begin, r_end) of the R_pad: block x covers rows r_begin + 32 x ..)
__global__ void k_upload_rowmajor(const float *__restrict__ x, int64_t R, int32_t C,
                                  int64_t R_pad, uint32_t *__restrict__ keys,
                                  int32_t *__restrict__ err, int64_t r_begin, int64_t r_end) {
  __shared__ uint32_t tile[32][33];
  const int64_t r0 = r_begin + (int64_t)blockIdx.x * 32;
  const int32_t c0 = blockIdx.y * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;
  bool bad = false;
#pragma unroll
  for (int j = ty; j < 32; j += 8) {
    const int64_t r = r0 + j;
    const int32_t c = c0 + tx;
    uint32_t k = 0u;
    if (r < R && c < C) {
      const uint32_t u = __float_as_uint(__ldg(x + r * C + c));
      bad |= not_finite(u);
      k = order_key(u);
    }
    tile[j][tx] = k;
  }
  if (__any_sync(0xFFFFFFFFu, bad) && (tx == 0)) atomicOr(err, 1);
  __syncthreads();
#pragma unroll
  for (int j = ty; j < 32; j += 8) {
    const int32_t c = c0 + j;
    const int64_t r = r0 + tx;
    if (c < C && r < r_end) keys[(int64_t)c * R_pad + r] = tile[tx][j];
  }
}

// Column-major x[C][R] -> keys[C][R_pad]: a block walks 4,096 rows of one column (blockIdx.y, and
// further columns gridDim.y apart), four rows per thread and step: one 16-byte load where every
// column starts on a 16-byte boundary (VEC), else four 4-byte loads a warp's width apart; keys are
// stored the same way.  Bound: HBM.  (One element per thread with its column found by a 64-bit
// division took 128 us at 33,333 x 777, now 40 us.)
constexpr int kColRows = 4096;

template <bool VEC>
__global__ void __launch_bounds__(256) k_upload_colmajor(const float *__restrict__ x, int64_t R,
                                                         int32_t C, int64_t R_pad,
                                                         uint32_t *__restrict__ keys,
                                                         int32_t *__restrict__ err) {
  const int64_t r_lo = (int64_t)blockIdx.x * kColRows;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  bool bad = false;
  for (int64_t c = blockIdx.y; c < C; c += gridDim.y) {
    const uint32_t *src = reinterpret_cast<const uint32_t *>(x) + c * R;
    uint32_t *dst = keys + c * R_pad;
#pragma unroll
    for (int k = 0; k < kColRows / 1024; ++k) {
      const int64_t r0 = r_lo + k * 1024 + warp * 128;  // the warp's 128 rows
      if (VEC) {
        const int64_t r = r0 + 4 * lane;
        if (r < R_pad) {  // (R_pad and R are multiples of 4)
          uint4 v = make_uint4(0u, 0u, 0u, 0u);
          if (r < R) {
            v = __ldg(reinterpret_cast<const uint4 *>(src + r));
            bad |= not_finite(v.x) || not_finite(v.y) || not_finite(v.z) || not_finite(v.w);
            v = make_uint4(order_key(v.x), order_key(v.y), order_key(v.z), order_key(v.w));
          }
          *reinterpret_cast<uint4 *>(dst + r) = v;
        }
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int64_t r = r0 + 32 * j + lane;
          if (r < R_pad) {
            uint32_t key = 0u;
            if (r < R) {
              const uint32_t u = __ldg(src + r);
              bad |= not_finite(u);
              key = order_key(u);
            }
            dst[r] = key;
          }
        }
      }
    }
  }
  if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicOr(err, 1);
}

// Pair bitmap: G[(a*C + b)*Wst + w] bit j = [key(32w+j, b) > key(32w+j, a)].
// A block covers 32 words (1024 rows) of kBW columns a (one per warp, its 1024 keys held in
// registers).  Each unordered pair a < b is compared once: the ballot of kb > ka gives G[a][b]
// and the ballot of kb < ka gives G[b][a] (ties set neither).  The b-columns of the chunk stream
// through a double-buffered shared-memory stage filled with cp.async, so their loads overlap
// the ballots; lane 0 parks the 32 ballots of a pair in shared memory and the warp then writes
// them as two coalesced 128-byte rows.  With few (chunk, a-block) pairs (small matrices), the
// stages of b-columns are also split across blockIdx.z (stage st goes to z = st mod gridDim.z),
// so the launch still fills the GPU and the long first a-blocks share their work.
constexpr int kBW = 8;  // warps (a-columns) per block
constexpr int kBS = 4;  // b-columns per stage

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  const unsigned saddr = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(saddr), "l"(gmem));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

__global__ void __launch_bounds__(kBW * 32, 4) k_build_bitmap(const uint32_t *__restrict__ keys,
                                                              int64_t R_pad, int32_t C,
                                                              int64_t Wst,
                                                              uint32_t *__restrict__ G) {
  __shared__ __align__(16) uint32_t sb[2][kBS][1024];
  __shared__ uint32_t s_out[kBW][2][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t w0 = (int64_t)blockIdx.x * 32;
  const int nw = (int)((Wst - w0 < 32) ? (Wst - w0) : 32);  // words of this chunk
  const int a0 = blockIdx.y * kBW;
  const int a = a0 + warp;
  const bool a_ok = a < C;
  uint32_t ka[32];
#pragma unroll
  for (int j = 0; j < 32; ++j)
    ka[j] = (a_ok && j < nw) ? __ldg(keys + (int64_t)a * R_pad + (w0 + j) * 32 + lane) : 0u;
  if (a_ok && lane < nw && blockIdx.z == 0) G[((int64_t)a * C + a) * Wst + w0 + lane] = 0u;
  const int bstart = a0 + 1;
  const int nstages = bstart < C ? (C - bstart + kBS - 1) / kBS : 0;
  const int S = (int)gridDim.z, z = (int)blockIdx.z;
  const int my_stages = nstages > z ? (nstages - z + S - 1) / S : 0;  // stages z, z + S, ...
  const int pieces = nw * 8;  // 16-byte pieces of one column's chunk
  auto issue = [&](int st, int buf) {
    const int b0 = bstart + st * kBS;
    for (int i = threadIdx.x; i < kBS * pieces; i += blockDim.x) {
      const int bb = i / pieces, piece = i - bb * pieces;
      const int b = b0 + bb;
      if (b < C)
        cp_async16(&sb[buf][bb][piece * 4], keys + (int64_t)b * R_pad + w0 * 32 + piece * 4);
    }
    cp_commit();
  };
  if (my_stages > 0) issue(z, 0);
  for (int k = 0; k < my_stages; ++k) {
    const int st = z + k * S;
    if (k + 1 < my_stages) {
      issue(st + S, (k + 1) & 1);
      cp_wait<1>();
    } else {
      cp_wait<0>();
    }
    __syncthreads();
    const int buf = k & 1, b0 = bstart + st * kBS;
    if (a_ok) {
      for (int bb = 0; bb < kBS; ++bb) {
        const int b = b0 + bb;
        if (b >= C) break;
        if (b <= a) continue;
        const uint32_t *col = sb[buf][bb];
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const uint32_t kb = col[j * 32 + lane];
          const uint32_t gt = __ballot_sync(0xFFFFFFFFu, kb > ka[j]);
          const uint32_t lt = __ballot_sync(0xFFFFFFFFu, kb < ka[j]);
          if (lane == 0) {
            s_out[warp][0][j] = gt;
            s_out[warp][1][j] = lt;
          }
        }
        __syncwarp();
        if (lane < nw) {
          G[((int64_t)a * C + b) * Wst + w0 + lane] = s_out[warp][0][lane];
          G[((int64_t)b * C + a) * Wst + w0 + lane] = s_out[warp][1][lane];
        }
        __syncwarp();
      }
    }
    __syncthreads();  // this buffer is consumed before it is refilled
  }
}

// Pair bitmap from the bit planes of the per-row rank codes (codes.cu): comparing codes is
// comparing keys (the codes keep every within-row order), and a word of planes holds one bit of
// 32 rows' codes, so one lane compares 32 rows at once.  Going from the lowest plane to the
// highest, with A and B the planes of columns a and b,
//   gt = (B & ~A) | (~(A ^ B) & gt)      lt = (A & ~B) | (~(A ^ B) & lt)
// (each one three-input logic instruction, lop3 with truth tables 0x8E and 0xB2) leave
// gt = [code_b > code_a] = G[a][b] and lt = [code_a > code_b] = G[b][a] in every bit: a higher
// differing bit overrides the lower ones, equal bits keep them.  Ties and pad rows (code 0
// everywhere) set neither.
// A warp owns two a-columns (their planes in registers) and one chunk of 64 words of rows (two
// words per lane, so every store is one coalesced 256-byte row piece), and walks b over a piece
// of consecutive columns after its own; the block's eight warps share the staged b planes.
// The row chunk is the fastest block index, so the blocks resident together write adjacent
// 256-byte pieces of the same pair rows, which L2 then merges into whole sectors before they
// reach DRAM.  The b-range of an a-block is cut into pieces of 16 << shift columns, so that the
// launch has enough blocks of about the same work to fill the GPU evenly (the first a-blocks
// pair with many more columns than the last ones): see launch_build_bitmap_planes.  The pieces
// run in the order of their first column (then of the a-block), so the blocks in flight together
// read the same b planes, which stay in L2 between them.
constexpr int kPA = 2;            // a-columns per warp
constexpr int kBuildWarps = 8;    // warps per block
constexpr int kABlock = kBuildWarps * kPA;  // a-columns per block
constexpr int kMaxPieceShift = 3;  // pieces of 16, 32, 64 or 128 columns
constexpr int kMaxABlocks = 1024 / kABlock;  // C <= 1,024
// pieces of 16 columns over every a-block of 16: 64 - g for a-block g
static_assert(kABlock == 16, "the piece count below");
constexpr int kMaxPieces = kMaxABlocks * (kMaxABlocks + 1) / 2;

struct PieceTable {
  uint16_t item[kMaxPieces];  // piece y of the launch: a-block << 8 | piece within the a-block
};

template <int LUT>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(d) : "r"(a), "r"(b), "r"(c), "n"(LUT));
  return d;
}

// The lowest plane, and one further plane's step, for both directions of a pair in the two words
// of a lane.
__device__ __forceinline__ void plane_first(uint2 A, uint2 B, uint2 &gt, uint2 &lt) {
  gt = make_uint2(B.x & ~A.x, B.y & ~A.y);
  lt = make_uint2(A.x & ~B.x, A.y & ~B.y);
}
__device__ __forceinline__ void plane_step(uint2 A, uint2 B, uint2 &gt, uint2 &lt) {
  gt.x = lop3<0x8E>(A.x, B.x, gt.x);  // (B & ~A) | (~(A ^ B) & gt)
  gt.y = lop3<0x8E>(A.y, B.y, gt.y);
  lt.x = lop3<0xB2>(A.x, B.x, lt.x);  // (A & ~B) | (~(A ^ B) & lt)
  lt.y = lop3<0xB2>(A.y, B.y, lt.y);
}

constexpr int kBB = 8;  // b-columns per staged batch (40 KB of static shared memory at NB = 10)

__device__ __forceinline__ void cp_async16_bm(void *smem, const void *gmem) {
  const unsigned saddr = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(saddr), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_commit_bm() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_wait_bm() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// The b planes of a block's piece are staged in shared memory, kBB columns at a time and
// double-buffered (cp.async by the whole block; the next batch is in flight while the current
// one is compared), so the eight warps share one copy.  A column's chunk is one contiguous span
// [NB][64] of the planes, copied as is; a lane reads the two words of a plane as one 8-byte load
// (a warp's loads are one 256-byte line: no bank conflicts).
// Two words per lane and two a-columns give eight independent comparator chains per b column
// within 80 registers (24 warps per SM), and everything a pair costs besides its comparators
// (addresses, stores, the warp sum of its counts) comes once per 64 words.
// The pair counts are accumulated too (cnt, zeroed beforehand): for a < b, cnt[a * C + b] holds
// the rows of G[a][b] (its popcount) in its low 32 bits and those of G[b][a] in its high 32
// bits.  Each warp adds its 64 words' counts of a pair by one warp sum (the two directions'
// counts packed in 16-bit halves, at most 2,048 each); lane j keeps the sums of the j-th of 32
// consecutive b columns, so that the atomics (64-bit) go out 32 at a time.
// What bounds it: the ALU pipe (40 lop3 of about 54 ALU instructions per pair and 64 words; the
// pipe is about 80% busy, the stores alone would take 1.25 ms at 60,000 x 1,000).  Measured with
// the planes' transposition, before (one word per lane, four a-columns per warp, planes written
// by the rank kernel) and now: 60,000 x 1,000 2.00 -> 1.65 ms, 33,333 x 777 685 -> 576 us,
// 20,000 x 500 185 -> 140 us, 10,000 x 100 44 -> 14 us.  Without the counts it takes 1.36 ms; four
// blocks per SM (64 registers, spills) 1.87 ms, four a-columns per warp (128 registers, two
// blocks) 1.83 ms, the b loop unrolled 2 or 4 times 1.71-1.73 ms.
// In the last chunk, words past Wst have zero planes in every column: they compare equal, so
// their words are zero (and not stored) and add nothing to the sums.
template <int NB>
__global__ void __launch_bounds__(kBuildWarps * 32, 3) k_build_bitmap_planes(const uint32_t *__restrict__ planes,
                                                             int32_t C, int64_t Wst,
                                                             int64_t chunks, int shift,
                                                             PieceTable tab,
                                                             uint32_t *__restrict__ G,
                                                             unsigned long long *__restrict__ cnt) {
  constexpr int kSpan = NB * 64;  // words of a column's chunk
  __shared__ __align__(16) uint32_t s_b[2][kBB][kSpan];
  // waits for the preceding kernel of a programmatic launch (the planes' and counts' writer)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // this block's a-block and piece (blockIdx.x is the row chunk: the blocks running together
  // write neighbouring pieces of the same pair rows)
  const int item = tab.item[blockIdx.y];
  const int ablk = item >> 8, piece = item & 0xFF;
  const int64_t ch = blockIdx.x;
  const int64_t w = ch * 64 + 2 * lane;  // the lane's words w, w + 1 (Wst is even: both or none)
  const bool w_ok = w < Wst;
  const int a0 = ablk * kABlock + warp * kPA;
  const int b_lo = ablk * kABlock + (piece << (shift + 4));  // the piece's b-range
  const int b_hi = min(C, b_lo + (16 << shift));
  const int b_first = max(b_lo, ablk * kABlock + kPA);  // the first b any warp of the block needs
  const int64_t cstride = chunks * kSpan;               // words between columns of the planes
  const uint32_t *pl = planes + ch * kSpan;             // column c's chunk at pl + c * cstride
  auto issue = [&](int t, int nbb) {  // batch t: columns b_first + t kBB + bb, bb < nbb
    const int bs = b_first + t * kBB;
    for (int j = threadIdx.x; j < nbb * (kSpan / 4); j += kBuildWarps * 32) {
      const int bb = j / (kSpan / 4), part = j - bb * (kSpan / 4);
      cp_async16_bm(&s_b[t & 1][bb][part * 4], pl + (int64_t)(bs + bb) * cstride + part * 4);
    }
    cp_commit_bm();
  };
  const int n_b = b_hi - b_first;  // (<= 0: no b beyond the block's columns in this piece)
  const int n_batches = n_b > 0 ? (n_b + kBB - 1) / kBB : 0;
  if (n_batches > 0) issue(0, min(kBB, n_b));
  uint2 A[kPA][NB];
#pragma unroll
  for (int i = 0; i < kPA; ++i) {
    const uint2 *src = reinterpret_cast<const uint2 *>(pl + (int64_t)(a0 + i) * cstride) + lane;
#pragma unroll
    for (int p = 0; p < NB; ++p) A[i][p] = a0 + i < C ? __ldg(src + 32 * p) : make_uint2(0u, 0u);
  }
  const int64_t row = (int64_t)C * Wst;  // words between G[a][.] and G[a + 1][.]
  // this warp's 64 words' counts of G[a][b] (gt) and G[b][a] (lt), packed, summed over the lanes
  auto warp_counts = [&](uint2 gt, uint2 lt) -> unsigned {
    return __reduce_add_sync(0xFFFFFFFFu,
                             (unsigned)(__popc(gt.x) + __popc(gt.y)) +
                                 ((unsigned)(__popc(lt.x) + __popc(lt.y)) << 16));
  };
  auto add_counts = [&](int a, int b, unsigned n) {  // (a < b)
    if (n)
      atomicAdd(cnt + (int64_t)a * C + b,
                (unsigned long long)(n & 0xFFFFu) | ((unsigned long long)(n >> 16) << 32));
  };
  auto store = [&](uint32_t *p, uint2 v) { __stcs(reinterpret_cast<uint2 *>(p), v); };
  if (piece == 0 && a0 < C) {
    // the diagonal words, and the pairs among the warp's own columns
#pragma unroll
    for (int i = 0; i < kPA; ++i) {
      const int a = a0 + i;
      if (a >= C) break;
      if (w_ok) store(G + (int64_t)a * row + (int64_t)a * Wst + w, make_uint2(0u, 0u));
#pragma unroll
      for (int i2 = i + 1; i2 < kPA; ++i2) {
        const int b = a0 + i2;
        if (b < C) {
          uint2 gt, lt;
          plane_first(A[i][0], A[i2][0], gt, lt);
#pragma unroll
          for (int p = 1; p < NB; ++p) plane_step(A[i][p], A[i2][p], gt, lt);
          if (w_ok) {
            store(G + (int64_t)a * row + (int64_t)b * Wst + w, gt);
            store(G + (int64_t)b * row + (int64_t)a * Wst + w, lt);
          }
          const unsigned n = warp_counts(gt, lt);
          if (lane == 0) add_counts(a, b, n);
        }
      }
    }
  }
  // G[a][b] at a * row + b * Wst, G[b][a] at b * row + a * Wst; (a + i)'s words sit i rows (or
  // i * Wst words) past a's: 32-bit offsets from two pointers (32-bit offsets for the b columns
  // too, from pointers set once per batch, made the build 5% slower)
  const uint32_t row32 = (uint32_t)row, wst32 = (uint32_t)Wst;  // (checked at launch)
  const bool active = a0 < C;  // (the whole warp; lanes past Wst store nothing)
  unsigned sum[kPA];
#pragma unroll
  for (int i = 0; i < kPA; ++i) sum[i] = 0u;
  for (int t = 0; t < n_batches; ++t) {
    if (t + 1 < n_batches) {
      issue(t + 1, min(kBB, n_b - (t + 1) * kBB));
      cp_wait_bm<1>();
    } else {
      cp_wait_bm<0>();
    }
    __syncthreads();  // batch t is in shared memory for every warp
    const int bs = b_first + t * kBB, nbb = min(kBB, b_hi - bs);
    const int bb0 = max(0, a0 + kPA - bs);  // the first b after the warp's own columns
    if (active && bb0 < nbb) {
      uint32_t *g_ab = G + (int64_t)a0 * row + (int64_t)(bs + bb0) * Wst + w;
      uint32_t *g_ba = G + (int64_t)(bs + bb0) * row + (int64_t)a0 * Wst + w;
#pragma unroll 1
      for (int bb = bb0; bb < nbb; ++bb) {
        const uint2 *sb = reinterpret_cast<const uint2 *>(&s_b[t & 1][bb][0]) + lane;
        uint2 gt[kPA], lt[kPA];
#pragma unroll
        for (int i = 0; i < kPA; ++i) plane_first(A[i][0], sb[0], gt[i], lt[i]);
#pragma unroll
        for (int p = 1; p < NB; ++p) {
          const uint2 B = sb[32 * p];
#pragma unroll
          for (int i = 0; i < kPA; ++i) plane_step(A[i][p], B, gt[i], lt[i]);
        }
        const bool mine = lane == ((t * kBB + bb) & 31);
#pragma unroll
        for (int i = 0; i < kPA; ++i) {
          if (w_ok) {
            store(g_ab + (uint32_t)i * row32, gt[i]);
            store(g_ba + (uint32_t)i * wst32, lt[i]);
          }
          const unsigned n = warp_counts(gt[i], lt[i]);
          sum[i] = mine ? n : sum[i];
        }
        g_ab += Wst;
        g_ba += row;
      }
    }
    if (active && ((t & 3) == 3 || t + 1 == n_batches)) {  // 32 columns' counts, or the last ones
      const int b = b_first + (t & ~3) * kBB + lane;
#pragma unroll
      for (int i = 0; i < kPA; ++i) {
        if (b < b_hi) add_counts(a0 + i, b, sum[i]);  // (0 where b is not after the columns)
        sum[i] = 0u;
      }
    }
    __syncthreads();  // every warp is done with this buffer before batch t + 2 refills it
  }
}

// Copies `total` pieces of pair rows without their padding: n of the `stride` pieces of each row (16
// bytes a piece, or 4 where the output starts between 16-byte boundaries), N pieces per thread, their
// loads ahead of their stores.  Bound: HBM.  33,333 x 777 (2.53 GB out): 0.72 ms, 3.5 TB/s written;
// the runtime's strided copy 1.29 ms, its plain copy of unpadded rows 0.75 ms.
template <class T, int N>
__global__ void __launch_bounds__(256) k_copy_rows(const T *__restrict__ G, int64_t stride,
                                                   uint32_t n, int64_t total,
                                                   T *__restrict__ out) {
  const int64_t q0 = (int64_t)blockIdx.x * (256 * N), r0 = q0 / n;
  const uint32_t c0 = (uint32_t)(q0 - r0 * n);
  T v[N];
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const uint32_t k = j * 256 + threadIdx.x, c = c0 + k, dr = c / n;
    if (q0 + k < total) v[j] = __ldcs(G + (r0 + dr) * stride + (c - dr * n));
  }
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const int64_t q = q0 + j * 256 + threadIdx.x;
    if (q < total) __stcs(out + q, v[j]);
  }
}

template <class T, int N>
cudaError_t copy_rows(const uint32_t *G, int64_t Gst, int64_t Wst, int64_t n_rows, uint32_t *out,
                      cudaStream_t s) {
  constexpr int kWords = sizeof(T) / 4, kBlock = 256 * N;
  const int64_t total = n_rows * (Wst / kWords), blocks = (total + kBlock - 1) / kBlock;
  if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
  k_copy_rows<T, N><<<(unsigned)blocks, 256, 0, s>>>(reinterpret_cast<const T *>(G), Gst / kWords,
                                                    (uint32_t)(Wst / kWords), total,
                                                    reinterpret_cast<T *>(out));
  return cudaGetLastError();
}

// Pairs of columns with equal values in some row: those whose two counts do not add up to R.
__global__ void __launch_bounds__(256) k_count_tied(const unsigned long long *__restrict__ cnt,
                                                    int32_t C, int64_t R, int32_t *out) {
  int n = 0;
  for (int64_t q = (int64_t)blockIdx.x * 256 + threadIdx.x; q < (int64_t)C * C;
       q += (int64_t)gridDim.x * 256) {
    const int64_t a = q / C, b = q - a * C;
    if (a < b) {
      const unsigned long long v = __ldg(cnt + q);
      n += (int64_t)(uint32_t)v + (int64_t)(v >> 32) != R;
    }
  }
  n = __reduce_add_sync(0xFFFFFFFFu, n);
  if (n && (threadIdx.x & 31) == 0) atomicAdd(out, n);
}

}  // namespace

cudaError_t launch_copy_rows(const uint32_t *G, int64_t Gst, int64_t Wst, int64_t n_rows,
                             uint32_t *out, cudaStream_t s) {
  return (reinterpret_cast<uintptr_t>(out) & 15) == 0
             ? copy_rows<uint4, 4>(G, Gst, Wst, n_rows, out, s)
             : copy_rows<uint32_t, 16>(G, Gst, Wst, n_rows, out, s);
}

cudaError_t launch_count_tied(const unsigned long long *cnt, int32_t C, int64_t R, int32_t *out,
                              cudaStream_t s) {
  const cudaError_t e = cudaMemsetAsync(out, 0, sizeof(int32_t), s);
  if (e != cudaSuccess) return e;
  const int64_t blocks = std::min<int64_t>(((int64_t)C * C + 255) / 256, 152 * 8);
  k_count_tied<<<(unsigned)blocks, 256, 0, s>>>(cnt, C, R, out);
  return cudaGetLastError();
}

cudaError_t launch_upload_rows(const float *x, int64_t R, int32_t C, int64_t R_pad,
                               uint32_t *keys, int32_t *err, int64_t r_begin, int64_t r_end,
                               cudaStream_t s) {
  if (r_begin < 0 || r_begin % 32 || r_end > R_pad || r_end % 32 || r_end <= r_begin)
    return cudaErrorInvalidValue;
  dim3 grid((unsigned)((r_end - r_begin) / 32), (unsigned)((C + 31) / 32));
  k_upload_rowmajor<<<grid, dim3(32, 8), 0, s>>>(x, R, C, R_pad, keys, err, r_begin, r_end);
  return cudaGetLastError();
}

cudaError_t launch_upload(const float *x, int64_t R, int32_t C, int64_t R_pad, int32_t layout,
                          uint32_t *keys, int32_t *err, cudaStream_t s) {
  if (layout == EBIC_LAYOUT_ROW_MAJOR) {
    return launch_upload_rows(x, R, C, R_pad, keys, err, 0, R_pad, s);
  } else {
    const dim3 grid((unsigned)((R_pad + kColRows - 1) / kColRows),
                    (unsigned)std::min<int32_t>(C, 65535));
    if (R % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0)
      k_upload_colmajor<true><<<grid, 256, 0, s>>>(x, R, C, R_pad, keys, err);
    else
      k_upload_colmajor<false><<<grid, 256, 0, s>>>(x, R, C, R_pad, keys, err);
  }
  return cudaGetLastError();
}

cudaError_t launch_build_bitmap(const uint32_t *keys, int64_t R_pad, int32_t C, int64_t Wst,
                                uint32_t *bitmap, cudaStream_t s) {
  const int64_t gx = (Wst + 31) / 32, gy = (C + kBW - 1) / kBW;
  // enough blocks for about four per SM, split over the b-stages of the first a-block at most
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    sms = 1;
  }
  const int64_t max_split = std::max<int64_t>(1, (C - 1 + kBS - 1) / kBS);
  const int64_t split =
      std::min<int64_t>(max_split, std::max<int64_t>(1, (4LL * sms + gx * gy - 1) / (gx * gy)));
  dim3 grid((unsigned)gx, (unsigned)gy, (unsigned)std::min<int64_t>(split, 65535));
  k_build_bitmap<<<grid, kBW * 32, 0, s>>>(keys, R_pad, C, Wst, bitmap);
  return cudaGetLastError();
}

cudaError_t launch_build_bitmap_planes(const uint32_t *planes, int32_t C, int64_t Wst,
                                       uint32_t *bitmap, unsigned long long *cnt, int num_sms,
                                       cudaStream_t s) {
  const int64_t chunks = code_plane_chunks(Wst);
  const int n_ablk = (C + kABlock - 1) / kABlock;
  if (!cnt) return cudaErrorInvalidValue;  // (the pair counts are always accumulated)
  // (the kernel offsets rows of the bitmap by up to C * Wst words in 32 bits)
  if (C < 2 || n_ablk > kMaxABlocks || chunks > 0x7FFFFFFF ||
      4 * (int64_t)C * Wst > (1ll << 32))
    return cudaErrorInvalidValue;
  // every (a-block g, piece p) with b in [16 g, C), in the order of the piece's first column
  // 16 g + len p, then of g.  The longest piece that still gives kWaves blocks per resident block
  // (three per SM), so that the last wave and the uneven first pieces are a small part of the launch
  // (8 waves against 24 and 60: 576, 599 and 598 us at 33,333 x 777; 1.64, 1.65 and 1.68 ms at
  // 60,000 x 1,000; with pieces of 128 columns always, a 10,000 x 100 matrix had 40 blocks)
  constexpr int64_t kWaves = 8;
  PieceTable tab{};
  int total = 0, shift = kMaxPieceShift;
  for (;; --shift) {
    const int len = 16 << shift;
    total = 0;
    for (int g = 0; g < n_ablk; ++g) total += (C - g * kABlock + len - 1) / len;
    if (shift == 0 || chunks * total >= kWaves * 3 * num_sms) break;
  }
  const int len = 16 << shift;
  int at = 0;
  for (int start = 0; start < C; start += std::min(len, kABlock))
    for (int g = 0; g < n_ablk && g * kABlock <= start; ++g)
      if ((start - g * kABlock) % len == 0)
        tab.item[at++] = (uint16_t)(g << 8 | (start - g * kABlock) / len);
  if (at != total) return cudaErrorInvalidValue;
  // (scheduled while the planes' kernel drains: rank codes, planes and build so launched: 59 to
  // 55 us for load, build and counts at 6,122 x 22, 63 to 59 at 3,000 x 200)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)chunks, (unsigned)total);
  cfg.blockDim = dim3(kBuildWarps * 32);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
#define EBIC_BUILD(NB) \
  case NB:             \
    return cudaLaunchKernelEx(&cfg, k_build_bitmap_planes<NB>, planes, C, Wst, chunks, shift, tab, \
                              bitmap, cnt)
  switch (code_plane_bits(C)) {
    EBIC_BUILD(1);
    EBIC_BUILD(2);
    EBIC_BUILD(3);
    EBIC_BUILD(4);
    EBIC_BUILD(5);
    EBIC_BUILD(6);
    EBIC_BUILD(7);
    EBIC_BUILD(8);
    EBIC_BUILD(9);
    EBIC_BUILD(10);
    default: return cudaErrorInvalidValue;
  }
#undef EBIC_BUILD
}
