// The stage kernel of the 58-variable formulations (ccz4_fo_*).
#ifndef CCZ4_FO_STAGE_CUH
#define CCZ4_FO_STAGE_CUH

#include "derive.h"
#include "fo_algebra.cuh"

#ifndef CCZ4_FO_MIN_BLOCKS
#define CCZ4_FO_MIN_BLOCKS 4
#endif

namespace ccz4 {

struct FoStageArgs {
  const double *U;  // U_n
  double *acc;      // RK accumulator
  double *out;      // plain right-hand side (MODE < 0), next stage state, or U_{n+1}
  double dt;
};

namespace {

// Receives d_t of each variable of one interior point and applies the stage
// update at once; the last stage holds g~ and A~ back for the enforcement.
template <int MODE>
struct FoSink {
  long long S, i;
  const FoStageArgs &a;
  double ug[6], uA[6];
  __device__ __forceinline__ void operator()(int v, double k) {
    const long long o = v * S + i;
    if (MODE < 0) {
      a.out[o] = k;
      return;
    }
    double acc = MODE == 0 ? 0.0 : a.acc[o];
    const double un = rk_combine<(MODE < 0 ? 0 : MODE), double>(a.U[o], acc, k, a.dt);
    if (MODE < 3) a.acc[o] = acc;
    if (MODE == 3 && v >= GXX && v <= GZZ) {
      ug[v - GXX] = un;
      return;
    }
    if (MODE == 3 && v >= AXX && v <= AZZ) {
      uA[v - AXX] = un;
      return;
    }
    a.out[o] = un;
  }
  __device__ __forceinline__ void finish() {
    if (MODE != 3) return;
    enforce_point<double>(ug, uA);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      a.out[(GXX + c) * S + i] = ug[c];
      a.out[(AXX + c) * S + i] = uA[c];
    }
  }
};

// One point's view of the state and of the derivative buffer (derive.h: slot
// 4 v + k the first-derivative sum of field v along axis k, 4 v + 3 its
// dissipation sum); the strides are the axes.
struct FoView {
  const double *c;   // field 0 of the state at the point
  const double *d;   // slot 0 at the point
  long long S, np;   // distance between fields of the state, between slots of the buffer
  int st[3];
};
template <class D>
__device__ __forceinline__ D ld(const FoView &N, int v, int) { return N.c[v * N.S]; }
template <class D>
__device__ __forceinline__ D fd1(const FoView &N, int v, int axis, const D &c1) {
  return __ldcs(N.d + (4 * v + axis) * N.np) * c1;
}
template <class D, class R>
__device__ __forceinline__ D d1u(const FoView &N, int v, int axis) { return __ldcs(N.d + (4 * v + axis) * N.np); }
template <class D>
__device__ __forceinline__ D ko_sum(const FoView &N, int v) { return __ldcs(N.d + (4 * v + 3) * N.np); }

__device__ __forceinline__ FoView fo_view(const GridView &g, const double *der, const double *in, long long i,
                                          long long q) {
  return FoView{in + i, der + q, g.S, (long long)g.wcap * (g.p * g.p * g.p), {0, 1, 2}};
}

// All variables of one Sommerfeld ghost cell: the radiative condition (Eq.
// exa_sommerfeld_inter) with the cell's static geometry, and the stage
// update.
template <int MODE>
__device__ __forceinline__ void fo_ghost_cell(const GridView &g, const ccz4_params &P, const double *__restrict__ in,
                                              const double *__restrict__ ini, const FoStageArgs &a, long long id) {
  const GhostGeo *gg = g.ghost_geo + id;
  const long long sn = __ldg(&gg->sn);
  if (sn < 0) return;
  const double geo = __ldg(&gg->geo), ir = __ldg(&gg->ir);
#pragma unroll 4
  for (int v = 0; v < NVF; ++v) {
    const double cv = v < NV ? P.somm_speed[v] : 1.0;
    const long long o = v * g.S + g.n_points + id;
    const double qg = __ldg(in + o);
    const double qn = __ldg(in + v * g.S + sn);
    const double k = -cv * geo * (qg - qn) - cv * ir * (qg - __ldg(ini + o));
    if (MODE < 0) {
      a.out[o] = k;
      continue;
    }
    double acc = MODE == 0 ? 0.0 : a.acc[o];
    const double un = rk_combine<(MODE < 0 ? 0 : MODE), double>(a.U[o], acc, k, a.dt);
    if (MODE < 3) a.acc[o] = acc;
    a.out[o] = un;
  }
}

// The first ghost_blocks blocks: one thread per ghost cell. The others: one
// thread per interior point of the window, the 58-variable right-hand side (RED: with the
// red terms; AUX: the auxiliary variables' equations too) from the derivative
// buffer and the stage update of what it evolves.
// The FP64 pipe holds it (ncu: 86 % busy; 3, 4 and 5 blocks within 1 %), so what
// counts is its FP64 operations: first differences unscaled, the terms of the
// D_kij equation with g~_ij under one coefficient, and the savings of
// ccz4_rhs_point took one step at 54^3 from 4.59 to 4.11 ms, at 90^3 from 18.8
// to 16.7 (reconstructed second order 13.1 to 12.0).
template <int MODE, bool RED, bool AUX>
__global__ void __launch_bounds__(128, CCZ4_FO_MIN_BLOCKS)
    fo_interior_kernel(GridView g, FoPhys F, StencilCoef<double> C, ccz4_params P, const double *__restrict__ der,
                       const double *__restrict__ in, const double *__restrict__ ini, FoStageArgs a, int ghost_blocks) {
  if ((int)blockIdx.x < ghost_blocks) {
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id < g.n_ghost) fo_ghost_cell<MODE>(g, P, in, ini, a, id);
    return;
  }
  const long long q = (long long)(blockIdx.x - ghost_blocks) * blockDim.x + threadIdx.x, p3 = g.p * g.p * g.p;
  if (q >= g.wn * p3) return;
  const long long i = g.w0 * p3 + q;
  const FoView N = fo_view(g, der, in, i, q);
  FoSink<MODE> sink{g.S, i, a};
  fo_rhs_point<RED, AUX>(F, N, C, sink);
  sink.finish();
}

inline StencilCoef<double> fo_coefs(double dx, double eps) {
  StencilCoef<double> C;
  C.c1 = 1.0 / (12.0 * dx);
  C.c2 = 1.0 / (12.0 * dx * dx);
  C.c3 = 1.0 / (144.0 * dx * dx);
  C.cko = eps / (64.0 * dx);
  return C;
}

// Launches the stage kernel of one (MODE, RED, AUX) on the interior points of the window and, with the first
// one, every ghost cell.
template <int MODE, bool RED, bool AUX>
cudaError_t launch_fo_interior(const GridView &g, const ccz4_params &P, const double *der, const double *in,
                               const double *ini, const FoStageArgs &a, cudaStream_t s) {
  const FoPhys F{make_phys<double>(P), P.mu};
  const long long points = (long long)g.wn * g.p * g.p * g.p, ghosts = g.w0 == 0 ? g.n_ghost : 0;
  const int t = points < 16LL * g.sms * 128 ? 32 : 128;  // a small grid spreads over the SMs in shares of 32 points
  const long long gb = (ghosts + t - 1) / t, nb = (points + t - 1) / t;
  if (gb + nb == 0) return cudaSuccess;
  fo_interior_kernel<MODE, RED, AUX><<<(unsigned)(gb + nb), t, 0, s>>>(g, F, fo_coefs(g.dx, P.ko_eps), P, der, in, ini, a,
                                                                       (int)gb);
  return cudaGetLastError();
}

}  // namespace
}  // namespace ccz4

#endif
