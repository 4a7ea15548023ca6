// Check of one individual of a caller's CSR population, by one warp, before any kernel indexes the
// matrix with it (eval.cu, noalloc.cu).
#pragma once

#include <stdint.h>

#include "../../include/ebic.h"

// Lane k holds columns k and k + 32 (sentinels that no column and no other lane's sentinel equals
// past the length).  Returns, in every lane, whether a column is out of range or repeated, the
// start below 0, or the length outside [2, 64].  *c0, *c1 receive the lane's columns.
__device__ __forceinline__ bool csr_bad(const int32_t *__restrict__ cols, int32_t s, int32_t e,
                                        int32_t C, int lane, int *c0, int *c1) {
  constexpr unsigned kAll = 0xFFFFFFFFu;
  const int64_t L = (int64_t)e - s;
  *c0 = -1 - lane;
  *c1 = -33 - lane;
  if (s < 0 || L < 2 || L > EBIC_MAX_LEN) return true;  // (warp-uniform: s, e are)
  const bool in0 = lane < L, in1 = lane + 32 < L;
  if (in0) *c0 = cols[s + lane];
  if (in1) *c1 = cols[s + 32 + lane];
  // (every lane takes part in each collective: none sits in a short-circuited operand)
  const unsigned m0 = __match_any_sync(kAll, *c0), m1 = __match_any_sync(kAll, *c1);
  bool bad = (in0 && (*c0 < 0 || *c0 >= C)) || (in1 && (*c1 < 0 || *c1 >= C));
  bad = bad || __popc(m0) > 1 || __popc(m1) > 1;
  if (L > 32) {  // (warp-uniform)
    for (int j = 0; j < 32; ++j) {
      const int b = __shfl_sync(kAll, *c0, j);
      bad = bad || *c1 == b;
    }
  }
  return __any_sync(kAll, bad);
}
