// A quotient in five FP64 operations, for kernels that the narrow FP64 pipe holds.
#pragma once

#include "fixed_stencil.cuh"

namespace ccz4 {

// num / den within an ulp, for a normal den below 2^1022, |num| of 2^-950 and more (or zero) and a normal
// quotient: the reciprocal of den's mantissa in FP32, its exponent put back by integer operations, gives r with
// an error below 2^-22.6; a step q <- q + r (num - den q), the residual correction of P. Markstein (IBM J. Res.
// Dev. 34, 1990), whose residual one FMA gives, multiplies the error of q by it, so two steps from q = num r
// leave the rounding of the last. Operands that are not finite give a result that is not.
__host__ __device__ __forceinline__ double quotient(double num, double den) {
  const uint64_t b = fx_bits(den);
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b, e = (hi >> 20) & 0x7FFu;
  const unsigned mb = 0x3F800000u | ((hi & 0xFFFFFu) << 3) | (lo >> 29);  // [1, 2)
#ifdef __CUDA_ARCH__
  const unsigned f = __float_as_uint(__frcp_rn(__uint_as_float(mb)));  // (1/2, 1]
#else
  float m;
  memcpy(&m, &mb, 4);
  m = 1.0f / m;
  unsigned f;
  memcpy(&f, &m, 4);
#endif
  const unsigned rh = (hi & 0x80000000u) | ((f >> 3) + ((1919u - e) << 20));
  const double r = fx_from_bits(((uint64_t)rh << 32) | (uint64_t)(f << 29));
  double q = num * r;
  q = fma(r, fma(-den, q, num), q);
  return fma(r, fma(-den, q, num), q);
}

}  // namespace ccz4
