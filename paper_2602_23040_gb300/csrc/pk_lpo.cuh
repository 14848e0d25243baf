// 8-bit codes of the low-precision proxy, for the encoder and for the gather
// that fake-quantises the masters.  FP32 steps in the order packuv.h
// states, without fused multiply-adds.
#pragma once
#include "pk_common.cuh"

namespace pk {

__device__ __forceinline__ uint32_t lpo_code(float x, float lo, float delta, float L) {
  const float u = floorf(__fadd_rn(__fdiv_rn(__fsub_rn(x, lo), delta), 0.5f));
  if (!(u >= 0.0f)) return 0u;
  if (u >= L) return (uint32_t)L;
  return (uint32_t)u;
}

// 1 / delta for lpo_codes4, NaN (no code is certain) for a step whose
// reciprocal loses precision.
__device__ __forceinline__ float lpo_rstep(float delta) {
  return delta > 1e-30f && delta < 1e30f ? __frcp_rn(delta) : __int_as_float(0x7fffffff);
}

// lpo_code of four values (0 where not live) by a multiplication with rd =
// 1 / delta where that is certain to give the same code: x - lo is the same
// value, the product lies within 2^-23 relative of the quotient and the sum
// within 2 x 2^-24, so a sum u further than 1e-6 (1 + u) from an integer
// has the quotient form's floor (below 0 either form's code is 0).  The
// division for the others: 2e-6 (1 + u) of the values at a code u, so 3 in
// 10,000 of the 8-bit channels' and, of the positions', 6.5 in 100 in the
// middle of their range -- some lane of nearly every warp.  The four run
// without a branch per value, and one test leaves to the division.
__device__ __forceinline__ void lpo_codes4(const float (&x)[4], uint32_t live, float lo, float delta, float rd,
                                           float L, uint32_t (&q)[4]) {
  uint32_t unsure = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float u = __fadd_rn(__fmul_rn(__fsub_rn(x[i], lo), rd), 0.5f), fl = floorf(u);
    const bool sure = fabsf(u - fl - 0.5f) < 0.5f - fmaf(1e-6f, u, 1e-6f);
    q[i] = (live >> i) & 1u ? __float2uint_rz(fminf(fl, L)) : 0u;   // a negative floor saturates to 0
    unsure |= sure ? 0u : 1u << i;
  }
  unsure &= live;
  if (unsure) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if ((unsure >> i) & 1u) q[i] = lpo_code(x[i], lo, delta, L);
  }
}

}  // namespace pk
