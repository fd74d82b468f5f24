// Top-list primitives shared by the selection kernels.
#pragma once
#include <climits>

#include "common.cuh"

namespace sp {

// Order-preserving 32-bit key of a float (larger float -> larger key; -0 is
// taken as +0); 0 is reserved for "no entry".
SP_DEVINL uint32_t fkey(float v) {
  const uint32_t u = __float_as_uint(v + 0.0f);
  return (u >> 31) ? ~u : (u | 0x80000000u);
}
// The key of a logit; a NaN ranks next to zero (its sign is the compiler's), or (pass_nan) is passed over.
SP_DEVINL uint32_t logit_key(float v, bool pass_nan) { return pass_nan && v != v ? 0u : fkey(v); }
SP_DEVINL float fkey_inv(uint32_t k) {
  if (k == 0u) return -INFINITY;
  return __uint_as_float((k >> 31) ? (k & 0x7FFFFFFFu) : ~k);
}

// Warp-wide selection of the best `per` of `tot` contiguous (value, index)
// entries (value desc, index asc), E entries per lane at most; every lane gets
// the result, best first.  Each pick is two redux.sync reductions: the largest
// key, then the smallest index holding it.
template <int GL, int E>
SP_DEVINL void warp_merge_lists(const float* vin, const int* iin, int tot, int per, float (&out_v)[GL],
                                int (&out_i)[GL]) {
  const int lane = threadIdx.x & 31;
  uint32_t key[E];
  int ei[E];
#pragma unroll
  for (int k = 0; k < E; ++k) {
    const int idx = lane + 32 * k;
    key[k] = 0u;
    ei[k] = INT_MAX;
    if (idx < tot) {
      ei[k] = iin[idx];
      if (ei[k] != INT_MAX) key[k] = fkey(vin[idx]);
    }
  }
#pragma unroll
  for (int r = 0; r < GL; ++r) {
    out_v[r] = -INFINITY;
    out_i[r] = INT_MAX;
    if (r < per) {
      uint32_t bk = key[0];
      int bi = ei[0];
#pragma unroll
      for (int k = 1; k < E; ++k)
        if (key[k] > bk || (key[k] == bk && ei[k] < bi)) { bk = key[k]; bi = ei[k]; }
      const uint32_t mk = __reduce_max_sync(0xffffffffu, bk);
      const int mi = (int)__reduce_min_sync(0xffffffffu, bk == mk ? (uint32_t)bi : 0x7fffffffu);
      out_v[r] = fkey_inv(mk);
      out_i[r] = mk ? mi : INT_MAX;
#pragma unroll
      for (int k = 0; k < E; ++k)
        if (ei[k] == mi) { key[k] = 0u; ei[k] = INT_MAX; }
    }
  }
}

}  // namespace sp
