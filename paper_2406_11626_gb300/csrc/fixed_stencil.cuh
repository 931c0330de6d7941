// FD4 stencil sums of FP64 values in 64-bit integers.
//
// The weights of every stencil used here are small integers (8 and 1; 16, 1
// and 30; 15, 6, 1 and 60), so a stencil sum of values held as integers of a
// common unit is exact. Each sum is rounded once, to the nearest FP64 number;
// an FP64 evaluation of the same stencil rounds every partial sum.
//
// The unit of a sum is 2^-56 of (the power of two of) the largest value that
// the sum itself has: the four neighbours of its axis for a first derivative,
// the centre too for a second, all 19 values for the dissipation. Values
// within a factor of sixteen of the largest are held exactly; of a smaller one
// the bits below the unit are dropped, toward zero, so that the sums keep the
// symmetries of FP64's: f -> -f and a reflection change the sign of a result and
// no bit, and zeros, of either sign, add nothing. A dropped bit costs up to 8
// (first derivative) or 16 (second) units; the rounding of an FP64 difference at
// the scale of the largest value costs as much as 8 of them. Where the largest
// value's biased exponent is FX_TOP or more (infinities and NaN too), or that of a
// sum not all of zeros is below FX_FLOOR, the point is evaluated in FP64.
//
// Against extended precision, field by field on the puncture and gauge-wave
// data, the root-mean-square error of the second derivatives and of the
// dissipation is a hundredth of FP64's and less, that of the first derivatives
// 0.47 to 0.96 of it.
//
// Why integers: this GPU's FP64 pipe issues 2 operations per clock per SM,
// the integer pipes 64 and more (measured: FP64 add, multiply and FMA 2, the
// integer-to-FP64 conversion 1.9, 64-bit integer add 58, logic and shift 60
// per clock per SM). An FP64 operation therefore costs as much as 32 integer
// instructions on pipes that the FP64 kernels leave idle; a value's conversion
// takes about 12 and the return to FP64 about 20.
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

// A zero that the compiler cannot move or foresee: what depends on it is not evaluated ahead of the
// branch it stands in.
__host__ __device__ __forceinline__ int here_zero() {
  int z = 0;
#ifdef __CUDA_ARCH__
  asm volatile("mov.u32 %0, 0;" : "=r"(z));
#endif
  return z;
}

// 8 (a1 - b1) - (a2 - b2): the first-derivative stencil of the values at +1, -1, +2, -2, all of them
// zero or within the integer range (not fx_wild).
__host__ __device__ __forceinline__ double fx_first_in(double a1, double b1, double a2, double b2) {
  const unsigned key = fx_max(fx_max(fx_key(a1), fx_key(b1)), fx_max(fx_key(a2), fx_key(b2)));
  const unsigned u = fx_unit(fx_max(key, FX_FLOOR << 21));  // shifts zeros out
  const int64_t d1 = fx_in(a1, u) - fx_in(b1, u), d2 = fx_in(a2, u) - fx_in(b2, u);
  return fx_out<4>(d1 * 8 - d2, u);
}
__host__ __device__ __forceinline__ bool fx_wild(double u) {
  const uint64_t b = fx_bits(u);
  const unsigned hi = (unsigned)(b >> 32) & 0x7FFFFFFFu;
  return hi - (FX_FLOOR << 20) >= (FX_TOP - FX_FLOOR) << 20 && (hi | (unsigned)b) != 0;
}
// The same of any values. (The compiler predicates the FP64 side: its operations take their slots of the
// FP64 pipe whether or not a thread needs them.)
__host__ __device__ __forceinline__ double fx_first(double a1, double b1, double a2, double b2) {
  const unsigned u = fx_unit(fx_max(fx_max(fx_key(a1), fx_key(b1)), fx_max(fx_key(a2), fx_key(b2))));
  return fx_outside(u) ? fma(8.0, a1 - b1, -(a2 - b2)) : fx_first_in(a1, b1, a2, b2);
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

// ---- sums of values that wait as words ------------------------------------------------
// The word of a value: its 57-bit mantissa, of a negative value the complement, so that an
// arithmetic shift drops bits toward zero once the sign is taken off (fx_shifted); its rank: 0 for
// zero, 1 for subnormal values (whose word has a leading one that is not theirs; units in the integer
// range shift all of it out), else the biased exponent plus one. Above FX_LAST the word is the value's bits.
constexpr unsigned FX_FIRST = FX_FLOOR + 1, FX_LAST = FX_TOP;
__host__ __device__ __forceinline__ int64_t fx_word(double u, unsigned &rank) {
  const uint64_t b = fx_bits(u);
  const unsigned hi = (unsigned)(b >> 32) & 0x7FFFFFFFu, any = hi | (unsigned)b;
  rank = (hi >> 20) + (any < 1u ? any : 1u);
  const uint64_t m = ((b << 4) & 0x00FFFFFFFFFFFFF0ull) | 0x0100000000000000ull;
  return rank > FX_LAST ? (int64_t)b : (int64_t)(m ^ (uint64_t)((int64_t)b >> 63));
}
__host__ __device__ __forceinline__ double fx_value(int64_t w, unsigned rank) {
  if (rank > FX_LAST) return fx_from_bits((uint64_t)w);
  const uint64_t n = (uint64_t)(w >> 63), a = (uint64_t)w ^ n;
  return fx_from_bits((n & 0x8000000000000000ull) | ((uint64_t)(rank ? rank - 1 : 0) << 52) |
                      ((a >> 4) & 0x000FFFFFFFFFFFFFull));
}
// x >> s, the sign for s > 63
__host__ __device__ __forceinline__ int64_t fx_sar(int64_t x, unsigned s) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
#else
  return x >> (s > 63 ? 63 : s);
#endif
}
// The value of word w in a unit s binades above its own, dropped bits truncated.
__host__ __device__ __forceinline__ int64_t fx_shifted(int64_t w, unsigned s) { return fx_sar(w, s) - (w >> 63); }
// x / 2^s, truncated
__host__ __device__ __forceinline__ int64_t fx_div2(int64_t x, unsigned s) {
  const int64_t n = x >> 63;
  return fx_sar(x + n, s) - n;
}
// v units (fx_out<K>) to the nearest FP64 number, ties to even: CVT by the conversion instruction, or
// else in integers (for a kernel whose other warps hold the FP64 pipe).
template <int K, bool CVT>
__host__ __device__ __forceinline__ double fx_return(int64_t v, unsigned unit) {
#ifdef __CUDA_ARCH__
  if constexpr (CVT) return fx_out_cvt<K>(v, unit);
#endif
  return fx_out<K, true>(v, unit);
}

// The stencil sums of fx_point in FP64. Inline: a call's registers would be its callee's choice.
template <bool SECOND, class E>
__host__ __device__ __forceinline__ void fx_point_fp64(const int64_t *w, const E *ex, const int (&st)[3], double *out) {
  const int z = here_zero();
  w += z;
  ex += z;
  const double c = fx_value(w[0], ex[0]);
  double s[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double p[3], m[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int o = (j + 1) * st[k];
      p[j] = fx_value(w[o], ex[o]);
      m[j] = fx_value(w[-o], ex[-o]);
      s[j] += p[j] + m[j];
    }
    out[k] = fma(8.0, p[0] - m[0], -(p[1] - m[1]));
    if (SECOND) out[4 + k] = fma(-30.0, c, fma(16.0, p[0] + m[0], -(p[1] + m[1])));
  }
  out[3] = fma(-60.0, c, fma(15.0, s[0], fma(-6.0, s[1], s[2])));
}

// The stencil sums of the point at w, ex (neighbours at multiples of st[k] along axis k): out[0..2]
// first derivatives, out[3] dissipation, out[4..6] pure second derivatives. The neighbours of an axis are
// brought to the unit of their own largest; their part of a second derivative and of the dissipation is
// truncated to the unit of that sum where that is larger. FIRST_CVT: first derivatives return as the others do,
// with CVT (for a pass that leaves the FP64 pipe idle).
// Magnitudes in units: 18 x 2^57 for a first, 64 x (2^57 - 1) for a second derivative; the dissipation
// 3 x + s3 - 60 c = 4 (x - 15 c) + (s3 - x), x the sum of 5 t1 - 2 t2 over the axes, whose parts stay below
// 57 x 2^57 and 48 x 2^57, is formed as it is or, where that is too large, as its quarter with the two bits
// below kept as one (they can only tell which side of a tie it is).
template <bool SECOND, bool CVT, bool FIRST_CVT = false, class E>
__host__ __device__ __forceinline__ void fx_point(const int64_t *w, const E *ex, const int (&st)[3], double *out) {
  const unsigned e0 = ex[0];
  unsigned ep[3][3], em[3][3], u[3], top = e0, low = e0 - 1u;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      ep[k][j] = ex[(j + 1) * st[k]];
      em[k][j] = ex[-(j + 1) * st[k]];
    }
    u[k] = fx_max(fx_max(ep[k][0], em[k][0]), fx_max(ep[k][1], em[k][1]));
    low = u[k] - 1u < low ? u[k] - 1u : low;  // (zeros do not count)
    top = fx_max(top, fx_max(u[k], fx_max(ep[k][2], em[k][2])));
    u[k] = fx_max(u[k], FX_FIRST);  // shifts zeros out
  }
  if (top == 0) {
#pragma unroll
    for (int q = 0; q < (SECOND ? 7 : 4); ++q) out[q] = 0.0;
    return;
  }
  if (top > FX_LAST || top < FX_FIRST || low < FX_FIRST - 1u) {
    fx_point_fp64<SECOND>(w, ex, st, out);
    return;
  }
  int64_t x = 0, s3 = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int s = st[k];
    const int64_t p1 = fx_shifted(w[s], u[k] - ep[k][0]), m1 = fx_shifted(w[-s], u[k] - em[k][0]);
    const int64_t p2 = fx_shifted(w[2 * s], u[k] - ep[k][1]), m2 = fx_shifted(w[-2 * s], u[k] - em[k][1]);
    const int64_t t1 = p1 + m1, t2 = p2 + m2;
    x += fx_div2(t1 * 5 - t2 * 2, top - u[k]);
    if (SECOND) {
      const unsigned v = fx_max(u[k], e0);
      const int64_t q = 2 * fx_shifted(w[0], v - e0);
      out[4 + k] = fx_return<5, CVT>(fx_div2(t1 * 16 - t2, v - u[k]) - q * 15, (v << 21) | FX_LOW);
    }
    const int64_t f = (p1 - m1) * 8 - (p2 - m2);
    const unsigned unit = (u[k] << 21) | FX_LOW;
    out[k] = FIRST_CVT ? fx_return<5, true>(f, unit) : fx_out<5>(f, unit);
    s3 += fx_shifted(w[3 * s], top - ep[k][2]) + fx_shifted(w[-3 * s], top - em[k][2]);
  }
  const int64_t y = x - 15 * fx_shifted(w[0], top - e0), r = s3 - x, v = y + (r >> 2);
  const bool whole = (uint64_t)(v + (1ll << 60)) < 1ull << 61;  // 4 y + r fits
  out[3] = fx_return<5, CVT>(whole ? y * 4 + r : v | ((r & 3) != 0), ((top + (whole ? 0u : 2u)) << 21) | FX_LOW);
}

// The first-derivative sum along stride s alone, as fx_point takes it.
template <class E>
__host__ __device__ __forceinline__ double fx_first_sum(const int64_t *w, const E *ex, int s) {
  const unsigned a = ex[s], b = ex[-s], c = ex[2 * s], d = ex[-2 * s];
  const unsigned u = fx_max(fx_max(a, b), fx_max(c, d));
  if (u > FX_LAST || u < FX_FIRST) {
    const int z = here_zero();
    w += z;
    ex += z;
    if (u == 0) return 0.0;
    return fma(8.0, fx_value(w[s], ex[s]) - fx_value(w[-s], ex[-s]),
               -(fx_value(w[2 * s], ex[2 * s]) - fx_value(w[-2 * s], ex[-2 * s])));
  }
  const int64_t p = fx_shifted(w[s], u - a) - fx_shifted(w[-s], u - b);
  const int64_t m = fx_shifted(w[2 * s], u - c) - fx_shifted(w[-2 * s], u - d);
  return fx_out<5>(p * 8 - m, (u << 21) | FX_LOW);
}

// The sums of fx_point from values on the host: the centre c and the neighbours p[k][j], m[k][j] at
// distance j + 1 along axis k; with D1 the first and with D2 the pure second derivatives.
template <bool D1, bool D2>
inline void fx_axes(double c, const double (&p)[3][3], const double (&m)[3][3], double *d1, double *d2, double &ko) {
  const int st[3] = {1, 4, 16};  // the multiples up to 3 of these are 18 different places around the centre
  int64_t w[2 * 48 + 1];
  unsigned e[2 * 48 + 1];
  w[48] = fx_word(c, e[48]);
  for (int k = 0; k < 3; ++k)
    for (int j = 0; j < 3; ++j) {
      const int o = (j + 1) * st[k];
      w[48 + o] = fx_word(p[k][j], e[48 + o]);
      w[48 - o] = fx_word(m[k][j], e[48 - o]);
    }
  double o[7];
  fx_point<D2, true>(w + 48, e + 48, st, o);
  for (int k = 0; k < 3; ++k) {
    if (D1) d1[k] = o[k];
    if (D2) d2[k] = o[4 + k];
  }
  ko = o[3];
}

}  // namespace ccz4
