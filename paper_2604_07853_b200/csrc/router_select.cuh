// Selection of one token's experts by one warp: top-k of its fp32 logits (descending, ties to the lower
// expert id) and the softmax over the selected ones.  Lane l holds experts l, l + 32, ... in v
// (-inf past E); PER = experts per lane, a compile-time bound so that the loops unroll to exactly the
// work the expert count needs.
#pragma once
#include <math.h>

#include "common.cuh"

namespace qarl {

template <int PER>
__device__ __forceinline__ void select_topk(const float (&v)[PER], int E, int k, int lane, int32_t* id_out, float* w_out) {
  uint32_t taken = 0;  // bit j: this lane's j-th expert was selected
  float sel = 0.0f;    // lane j < k ends up holding the j-th selected logit
  int sel_id = 0;
  for (int r = 0; r < k; ++r) {
    float best = -INFINITY;
    int best_e = 0x7FFFFFFF;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      if (!((taken >> j) & 1u)) {
        const int e = lane + 32 * j;
        if (e < E && (v[j] > best || best_e == 0x7FFFFFFF)) {  // ascending e within a lane: strict > keeps the lower id
          best = v[j];
          best_e = e;
        }
      }
    }
    // Warp arg-max in two reductions instead of a five-step butterfly on (value, id) pairs: the largest
    // value through an order-preserving map of its bits to unsigned (-0 first folded onto +0, so equal
    // values map to equal keys), then the lowest id among the lanes that hold it.
    const uint32_t bits = __float_as_uint(best + 0.0f);
    const uint32_t key = best_e == 0x7FFFFFFF ? 0u : ((bits & 0x80000000u) ? ~bits : (bits | 0x80000000u));
    const uint32_t top = __reduce_max_sync(0xFFFFFFFFu, key);
    const int win_e = static_cast<int>(__reduce_min_sync(0xFFFFFFFFu, key == top ? static_cast<uint32_t>(best_e) : 0x7FFFFFFFu));
    const float win = __shfl_sync(0xFFFFFFFFu, best, win_e & 31);
    best = win;
    best_e = win_e;
    if ((best_e & 31) == lane) taken |= 1u << (best_e >> 5);
    if (lane == r) {
      sel = best;
      sel_id = best_e;
    }
  }
  // softmax over the k selected logits, in double: exp(l - max) / sum, rounded to fp32
  const double mx = static_cast<double>(__shfl_sync(0xFFFFFFFFu, sel, 0));
  double ex = lane < k ? exp(static_cast<double>(sel) - mx) : 0.0;
  double den = 0.0;  // summed in selection order (the one-launch router adds them as it selects)
  for (int j = 0; j < k; ++j) den += __shfl_sync(0xFFFFFFFFu, ex, j);
  if (lane < k) {
    id_out[lane] = sel_id;
    w_out[lane] = static_cast<float>(ex / den);
  }
}

}  // namespace qarl
