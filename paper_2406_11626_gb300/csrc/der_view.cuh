// One point's view of what the derivative pass wrote (derive.h), for the
// pointwise kernels: the algebra of a stage and the monitors.
#pragma once

#include "ccz4_algebra.cuh"
#include "derive.h"

// Loads of the derivative buffer, each value once: streaming; a translation
// unit whose kernel writes the buffer itself before reading it defines this
// as a coherent load before including.
#ifndef CCZ4_DER_LOAD
#define CCZ4_DER_LOAD __ldcs
#endif

namespace ccz4 {
namespace {

// One point's view of the derivative buffer, in place of the halo'd
// neighbourhood: the stencil values that ccz4_rhs_point asks for by field and
// stride are looked up in the slots of the derivative pass. The strides are
// those of the axes (0, 1, 2), nothing else is addressed with them.
template <bool MIXED>
struct DerView {
  const double *c;     // field 0 of the state at the point
  long long fs;        // distance between fields
  int st[3];
  const double *d;     // FP64 slots at the point
  const float *f;      // FP32 slots (mixed precision)
  const double *mix;
  const float *mixf;
  long long np, dnp;   // distance between slots of mix and of the derivative buffer
  __device__ __forceinline__ double at(int v, int) const { return c[v * fs]; }
  __device__ __forceinline__ double slot(int k) const { return CCZ4_DER_LOAD(d + k * dnp); }
  __device__ __forceinline__ float slotf(int k) const { return CCZ4_DER_LOAD(f + k * dnp); }
  __device__ __forceinline__ double mixed(int k) const { return CCZ4_DER_LOAD(mix + k * np); }
  __device__ __forceinline__ float mixedf(int k) const { return CCZ4_DER_LOAD(mixf + k * np); }
  // first-derivative sum along axis k, dissipation sum (k = 3) and pure second sum of field v
  __device__ __forceinline__ double fp64(int v, int k) const { return slot(MIXED ? (v == ALPHA ? 0 : 7) + k : 4 * v + k); }
  __device__ __forceinline__ double pure64(int v, int k) const {
    return slot(MIXED ? (v == ALPHA ? 4 : 11) + k : 4 * NV + 3 * der_second(v) + k);
  }
  __device__ __forceinline__ float fp32(int v, int k) const { return slotf(4 * der_f(v) + k); }
  __device__ __forceinline__ float pure32(int v, int k) const { return slotf(DER_F + 3 * der_f2(v) + k); }
};

template <class D, bool M>
__device__ __forceinline__ D ld(const DerView<M> &N, int v, int) { return N.c[v * N.fs]; }
template <class R, bool M>
__device__ __forceinline__ void ld2(const DerView<M> &N, int v, int, R &h, R &l) {
  const double u = N.c[v * N.fs];
  h = cvt<R>(u);
  l = cvt<R>(u - cvt<double>(h));
}
template <class D, class R, bool M>
__device__ __forceinline__ R centre(const DerView<M> &N, int v) { return cvt<R>(N.c[v * N.fs]); }
template <class D, bool M>
__device__ __forceinline__ D fd1(const DerView<M> &N, int v, int axis, const D &c1) { return N.fp64(v, axis) * c1; }
template <class D, class R, bool M>
__device__ __forceinline__ R d1u(const DerView<M> &N, int v, int axis) {
  if constexpr (M) return N.fp32(v, axis);
  else return N.fp64(v, axis);
}
template <class D, class R, bool M>
__device__ __forceinline__ R d1o(const DerView<M> &N, int v, int axis, const R &c1) { return d1u<D, R>(N, v, axis) * c1; }
template <class D, class R, bool M>
__device__ __forceinline__ R kosum(const DerView<M> &N, int v) { return d1u<D, R>(N, v, 3); }
template <class D, class O, bool SCALED = true, bool M>
__device__ __forceinline__ void second_ko(const DerView<M> &N, int v, const StencilCoef<D> &C, const StencilCoef<O> &,
                                          O dd[6], D &ko) {
  const int m = mix_slot(v);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int q = k == 0 ? 0 : k == 1 ? 3 : 5;
    dd[q] = N.pure64(v, k);
    if constexpr (SCALED) dd[q] = dd[q] * C.c2;
  }
  dd[1] = N.mixed(m);
  dd[2] = N.mixed(m + 1);
  dd[4] = N.mixed(m + 2);
  ko = N.fp64(v, 3);
}
template <class D, class R, bool SCALED, bool M>
__device__ __forceinline__ void second_sp(const DerView<M> &N, int v, const StencilCoef<D> &C, const StencilCoef<R> &CR,
                                          R dd[6], R &ko) {
  if constexpr (!M) {
    second_ko<D, R, SCALED>(N, v, C, CR, dd, ko);
  } else {
    const int m = mix_fslot(mix_slot(v));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int q = k == 0 ? 0 : k == 1 ? 3 : 5;
      dd[q] = N.pure32(v, k);
      if constexpr (SCALED) dd[q] = dd[q] * CR.c2;
    }
    dd[1] = N.mixedf(m);
    dd[2] = N.mixedf(m + 1);
    dd[4] = N.mixedf(m + 2);
    ko = N.fp32(v, 3);
  }
}
// second derivative d_k d_l (k, l known at compile time after unrolling)
template <class D>
__device__ __forceinline__ D fdkl(const DerView<false> &N, int v, int k, int l, const StencilCoef<D> &C) {
  if (k == l) return N.pure64(v, k) * C.c2;
  return N.mixed(mix_slot(v) + k + l - 1);
}

// The view of interior point i, its values from the state-shaped buffer `in`, its sums at place q of the
// derivative buffer.
template <bool M>
__device__ __forceinline__ DerView<M> der_view(const GridView &g, const double *der, const double *mix, const double *in,
                                               long long i, long long q) {
  DerView<M> N;
  N.c = in + i;
  N.fs = g.S;
  N.st[0] = 0;
  N.st[1] = 1;
  N.st[2] = 2;
  N.dnp = (long long)g.wcap * (g.p * g.p * g.p);
  N.d = der + q;
  N.f = reinterpret_cast<const float *>(der + DER_D * N.dnp) + q;
  N.mix = mix + i;
  N.mixf = reinterpret_cast<const float *>(mix) + i;
  N.np = g.n_points;
  return N;
}

}  // namespace
}  // namespace ccz4
