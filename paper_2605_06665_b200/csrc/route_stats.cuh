// Statistics of a router pass (tokens and summed scores per expert), shared by the router kernels of the bf16 mode.
#pragma once

#include "common.cuh"

namespace unipool {

// Counts are integers, and a block's score sums are rounded to multiples of 2^-28 and added as 64-bit integers too: the
// totals do not depend on the order in which the blocks arrive.  The accumulators start at zero and are left at zero.
struct RouteTotals {
  int32_t* counts_out; float* sum_out;
  int32_t* acc_counts; long long* acc_sums;
  uint32_t* ticket;                            // [0] blocks done, [1] a sum is not finite or out of range
};

// One block's share of expert i.  All scores of a call have one sign, so that an overflow of the total is seen by the block
// whose sum causes it, whatever the order; only sums that could add up that far read the total back.
__device__ __forceinline__ void add_route_total(const RouteTotals& r, int i, int count, float sum) {
  constexpr float kRange = 3.0e10f;            // below 2^35: a sum's multiple of 2^-28 fits 64 bits
  if (count != 0) atomicAdd(&r.acc_counts[i], count);
  if (!(fabsf(sum) < kRange)) {
    atomicOr(r.ticket + 1, 1u);
  } else if (sum != 0.f) {
    const long long v = __float2ll_rn(sum * 268435456.f);
    auto acc = reinterpret_cast<unsigned long long*>(&r.acc_sums[i]);
    if (fabsf(sum) * (float)gridDim.x < kRange) {
      atomicAdd(acc, (unsigned long long)v);
    } else {
      const long long was = (long long)atomicAdd(acc, (unsigned long long)v);
      const long long now = (long long)((unsigned long long)was + (unsigned long long)v);
      if (((was ^ now) & (v ^ now)) < 0) atomicOr(r.ticket + 1, 1u);
    }
  }
}

// What the block that arrives last does for every expert i, then for the ticket.
__device__ __forceinline__ void publish_route_total(const RouteTotals& r, int i, bool bad) {
  r.counts_out[i] = __ldcg(&r.acc_counts[i]);
  const long long fixed = __ldcg(&r.acc_sums[i]);
  r.sum_out[i] = bad ? __int_as_float(0x7fc00000) : (float)((double)fixed * (1.0 / 268435456.0));
  r.acc_counts[i] = 0;
  r.acc_sums[i] = 0;
}

// Sums v[i] over the lanes by recursive halving; lane l is left with value l in v[0].
__device__ __forceinline__ void sum_over_lanes(float (&v)[32], int lane) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    const bool upper = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < o; ++j) {
      const float send = upper ? v[j] : v[j + o], keep = upper ? v[j + o] : v[j];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
}

}  // namespace unipool
