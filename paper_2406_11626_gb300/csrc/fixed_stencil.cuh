// FD4 stencil sums of FP64 values in 64-bit integers.
//
// The weights of every stencil used here are small integers (8 and 1; 16, 1
// and 30; 15, 6, 1 and 60), so a stencil sum of values held as integers of a
// common unit is exact. The values of one stencil are brought to the unit
// 2^(e - 56), e the exponent of the largest of them: each is shifted right by
// its distance from e, which is exact for values within a factor of sixteen of
// the largest and otherwise drops bits below 2^-56 of it. The weights of the
// first derivative add up to 18, so its sum stays within 63 bits; those of the
// second derivative and of the dissipation over three axes add up to 64 and
// 192, so their partial sums drop two bits first (none is set while the
// values lie within a factor of four). Each sum is rounded once, to the
// nearest FP64 number. An FP64 evaluation of the same stencil rounds every
// partial sum, at the scale of the largest one: against extended precision on
// the puncture and gauge-wave data the second derivatives and the dissipation
// come out 10 to 100 times closer, the first derivatives as close or closer.
//
// Why integers: this GPU's FP64 pipe issues 2 operations per clock per SM,
// the integer pipes 64 and more (measured: FP64 add, multiply and FMA 2, the
// integer-to-FP64 conversion 1.9, 64-bit integer add 58, logic and shift 60
// per clock per SM). An FP64 operation therefore costs as much as 32 integer
// instructions on pipes that the FP64 kernels leave idle; a value's conversion
// takes about 12 and the return to FP64 about 20.
//
// A stencil whose largest value has a biased exponent of FX_TOP or more
// (infinities and NaN too) or below FX_FLOOR is evaluated in FP64.
#pragma once

#include <stdint.h>
#include <string.h>

namespace ccz4 {

// Below FX_FLOOR a result could leave the normal range, and zero would have to be told from the
// smallest values; from FX_TOP on a result could overflow.
constexpr unsigned FX_FLOOR = 72;
constexpr unsigned FX_TOP = 2030;
constexpr unsigned FX_LOW = 0x1FFFFFu;

__host__ __device__ __forceinline__ uint64_t fx_bits(double u) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(u);
#else
  uint64_t b;
  memcpy(&b, &u, 8);
  return b;
#endif
}
__host__ __device__ __forceinline__ double fx_from_bits(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double u;
  memcpy(&u, &b, 8);
  return u;
#endif
}
// The high word without its sign: ordered like the magnitude, the exponent in its top 11 bits.
__host__ __device__ __forceinline__ unsigned fx_key(double u) { return (unsigned)(fx_bits(u) >> 32) << 1; }
__host__ __device__ __forceinline__ unsigned fx_max(unsigned a, unsigned b) { return a > b ? a : b; }
// The key of a stencil's unit from the largest key of its values: its exponent, the bits below it set.
__host__ __device__ __forceinline__ unsigned fx_unit(unsigned key) { return key | FX_LOW; }
__host__ __device__ __forceinline__ bool fx_outside(unsigned unit) {
  return (unit >> 21) - FX_FLOOR >= FX_TOP - FX_FLOOR;
}

// x >> s, 0 for s > 63 (as the hardware shifts)
__host__ __device__ __forceinline__ uint64_t fx_shr(uint64_t x, unsigned s) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
#else
  return s > 63 ? 0 : x >> s;
#endif
}

// u in units of 2^(e - 1079), e the biased exponent of `unit`, dropped bits truncated
__host__ __device__ __forceinline__ int64_t fx_in(double u, unsigned unit) {
  const uint64_t b = fx_bits(u);
  const unsigned s = (unit - ((unsigned)(b >> 32) << 1)) >> 21;  // e - exponent of u
  const uint64_t m = ((b << 4) & 0x00FFFFFFFFFFFFFFull) | 0x0100000000000000ull;
  const uint64_t a = fx_shr(m, s), n = (uint64_t)((int64_t)b >> 63);
  return (int64_t)((a ^ n) - n);
}

// v units of 2^(e - 1075 - K) as FP64, rounded to nearest (ties away from zero; EVEN: to even, as the
// conversion instruction rounds)
template <int K, bool EVEN = false>
__host__ __device__ __forceinline__ double fx_out(int64_t v, unsigned unit) {
  const uint64_t n = (uint64_t)(v >> 63), a = ((uint64_t)v ^ n) - n;
#ifdef __CUDA_ARCH__
  const int z = __clzll((long long)a);
#else
  const int z = a ? __builtin_clzll(a) : 64;
#endif
  const uint64_t t = a << (z & 63);                 // top bit set (0 for v = 0)
  const unsigned up = EVEN && (t & 0x3FFu) == 0 ? (unsigned)(t >> 11) & 1u : 1u;
  const uint64_t r = (t >> 11) + ((unsigned)(t >> 10) & up);  // 53 bits, a carry goes into the exponent
  const uint64_t e = (uint64_t)((unit >> 21) + 10u - K - (unsigned)z) << 52;
  const uint64_t w = ((n & 0x8000000000000000ull) | e) + r;
  return a ? fx_from_bits(w) : 0.0;
}

#ifdef __CUDACC__
// The same by the conversion instruction, which runs on the FP64 pipe (one of
// its slots instead of about 20 integer instructions): to nearest, ties to even.
template <int K>
__device__ __forceinline__ double fx_out_cvt(long long v, unsigned unit) {
  const double d = __ll2double_rn(v);
  const int hi = __double2hiint(d) + (int)(((unit >> 21) - (1075u + K)) << 20);
  return v ? __hiloint2double(hi, __double2loint(d)) : 0.0;
}
#endif

// 8 (a1 - b1) - (a2 - b2): the first-derivative stencil of the values at +1, -1, +2, -2
__host__ __device__ __forceinline__ double fx_first(double a1, double b1, double a2, double b2) {
  const unsigned u = fx_unit(fx_max(fx_max(fx_key(a1), fx_key(b1)), fx_max(fx_key(a2), fx_key(b2))));
  if (fx_outside(u)) return fma(8.0, a1 - b1, -(a2 - b2));
  const int64_t d1 = fx_in(a1, u) - fx_in(b1, u), d2 = fx_in(a2, u) - fx_in(b2, u);
  return fx_out<4>(d1 * 8 - d2, u);
}

// The FP64 side of fx_laplacian: out of line, or the compiler evaluates it ahead of the branch.
__host__ __device__ __noinline__ inline double fx_laplacian_fp64(double c, double a, double b, double d, double e, double f,
                                                          double g) {
  return fma(-6.0, c, ((a + b) + (d + e)) + (f + g));
}

// The sum of the six values v minus 6 c (the 7-point Laplacian without 1 / h^2).
__host__ __device__ __forceinline__ double fx_laplacian(double c, const double (&v)[6]) {
  unsigned key = fx_key(c);
#pragma unroll
  for (int k = 0; k < 6; ++k) key = fx_max(key, fx_key(v[k]));
  const unsigned u = fx_unit(key);
  if (fx_outside(u)) return fx_laplacian_fp64(c, v[0], v[1], v[2], v[3], v[4], v[5]);
  int64_t s = fx_in(c, u) * -6;
#pragma unroll
  for (int k = 0; k < 6; ++k) s += fx_in(v[k], u);
  return fx_out<4>(s, u);
}

// From the centre c and the neighbours p[k][j], m[k][j] at distance j + 1 along
// axis k: the dissipation sum (over j of 15, -6, 1 times the sums of the six
// neighbours, minus 60 c); with D1 the first-derivative sums and with D2 the
// pure second-derivative sums 16 (p + m) - (p2 + m2) - 30 c of each axis.
template <bool D1, bool D2>
__host__ __device__ __forceinline__ void fx_axes(double c, const double (&p)[3][3], const double (&m)[3][3], double *d1,
                                                 double *d2, double &ko) {
  unsigned key = fx_key(c);
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int j = 0; j < 3; ++j) key = fx_max(key, fx_max(fx_key(p[k][j]), fx_key(m[k][j])));
  const unsigned u = fx_unit(key);
  if (fx_outside(u)) {
    double s[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (D1) d1[k] = fma(8.0, p[k][0] - m[k][0], -(p[k][1] - m[k][1]));
      if (D2) d2[k] = fma(-30.0, c, fma(16.0, p[k][0] + m[k][0], -(p[k][1] + m[k][1])));
#pragma unroll
      for (int j = 0; j < 3; ++j) s[j] += p[k][j] + m[k][j];
    }
    ko = fma(-60.0, c, fma(15.0, s[0], fma(-6.0, s[1], s[2])));
    return;
  }
  const int64_t q = fx_in(c, u) >> 2;
  int64_t s1 = 0, s2 = 0, s3 = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int64_t p1 = fx_in(p[k][0], u), m1 = fx_in(m[k][0], u), p2 = fx_in(p[k][1], u), m2 = fx_in(m[k][1], u);
    const int64_t t1 = p1 + m1, t2 = p2 + m2;
    if (D1) d1[k] = fx_out<4>((p1 - m1) * 8 - (p2 - m2), u);
    if (D2) d2[k] = fx_out<2>(((t1 >> 2) - 2 * q) * 16 - (t2 >> 2) + 2 * q, u);
    s1 += t1;
    s2 += t2;
    s3 += fx_in(p[k][2], u) + fx_in(m[k][2], u);
  }
  ko = fx_out<2>((((s1 >> 2) - 4 * q) * 5 - 2 * (s2 >> 2)) * 3 + (s3 >> 2), u);
}

}  // namespace ccz4
