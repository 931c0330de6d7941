// Right-hand side and fused RK4 stage kernels (templates; rhs.cu
// instantiates them for a single level, rhs_mesh.cu for refined meshes, so
// the two sets compile in parallel).
//
// algebra_kernel: one thread per interior point takes the point's values from
// the state, its stencil sums and mixed derivatives from the derivative pass
// (derive.cuh), evaluates the CCZ4 right-hand side plus Kreiss-Oliger
// dissipation, and either stores it (plain RHS) or applies the RK4 stage
// update in the same pass, so the right-hand side never travels through HBM.
// The last stage also enforces the algebraic constraints on the new state. R
// is the type of the pointwise algebra (double: FP64 path; float: mixed
// path). On a refined mesh each thread takes the stencil coefficients of its
// patch's level.
// Its first blocks advance the evolved Sommerfeld ghost cells (Eq.
// exa_sommerfeld_inter; the ghost shell of level 0), one thread per cell, in
// FP64 with no enforcement: they wait on memory while the interior points
// hold the FP64 pipe.
#pragma once

#include "ccz4_algebra.cuh"
#include "der_view.cuh"
#include "derive.cuh"

// Minimum resident blocks of 128 threads per SM requested for the algebra
// kernel. FP64: the FP64 pipe holds it (ncu: 91 % busy) at any of 3, 4 or 5
// blocks (36.81, 37.00, 36.53 ms per RK4 step at 144^3); mixed: the latency of
// its loads holds it and more warps hide more of it (17.13, 16.12, 15.83 ms).
#ifndef CCZ4_INTERIOR_MIN_BLOCKS
#define CCZ4_INTERIOR_MIN_BLOCKS 5
#endif
#ifndef CCZ4_INTERIOR_MIN_BLOCKS_MIXED
#define CCZ4_INTERIOR_MIN_BLOCKS_MIXED 5
#endif
// The last stage's enforcement reads the new g~ and A~ back from the output
// (written there as soon as they are known, by the same thread) instead of
// holding them in registers through the rest of the right-hand side, which
// frees 12 registers for the algebra. 0: hold them.
#ifndef CCZ4_ENFORCE_RELOAD
#define CCZ4_ENFORCE_RELOAD 1
#endif

// State, accumulator and output of the stage update: streaming
// (evict-first) loads and stores, each value is touched once, which leaves
// L2 to the kernel's register spills; 0 for plain ones.
#ifndef CCZ4_STAGE_STREAM
#define CCZ4_STAGE_STREAM 1
#endif

namespace ccz4 {

__device__ __forceinline__ double st_ld(const double *p) {
#if CCZ4_STAGE_STREAM
  return __ldcs(p);
#else
  return *p;
#endif
}
__device__ __forceinline__ void st_st(double *p, double v) {
#if CCZ4_STAGE_STREAM
  __stcs(p, v);
#else
  *p = v;
#endif
}

struct StageArgs {
  const double *U;  // U_n
  double *acc;      // RK accumulator
  double *out;      // plain RHS (MODE < 0), next stage state, or U_{n+1}
  double dt;
};


// Stencil coefficients of every level, in the differencing type (double)
// and in the algebra type R.
template <class R>
struct LevelCoef {
  StencilCoef<double> C[MAX_LEVELS];
  StencilCoef<R> CR[MAX_LEVELS];
};

// What a stage reads and writes besides the parameters.
struct StageBufs {
  const double *der;   // derivative buffer
  const double *mix;   // mixed second derivatives
  const double *in;    // the stage's input state
  const double *ini;   // initial values (ghost cells)
};

// Flat launches of the algebra kernel in the shapes other than the default
// (one resident block more or fewer, CCZ4_STAGE_SHAPE_*), RK4 stages 0..3
// only; instantiated in rhs_shapes.cu (single level) and rhs_mesh_shapes.cu.
cudaError_t launch_shaped_uniform(const GridView &g, int stage, const ccz4_params &P, const StageBufs &b,
                                  const StageArgs &a, cudaStream_t s);
cudaError_t launch_shaped_mesh(const GridView &g, int stage, const ccz4_params &P, const StageBufs &b,
                               const StageArgs &a, cudaStream_t s);

// Launches stage `stage` (-1: plain RHS) with the kernels of a single level
// (rhs.cu) or of a refined mesh (rhs_mesh.cu).
cudaError_t launch_stage_uniform(const GridView &g, const ccz4_params &P, int stage, const StageBufs &b,
                                 const StageArgs &a, cudaStream_t s);
cudaError_t launch_stage_mesh(const GridView &g, const ccz4_params &P, int stage, const StageBufs &b,
                              const StageArgs &a, cudaStream_t s);

namespace {


// Receives d_t Q_v of one interior point field by field and applies the
// stage update at once, so finished values leave the registers early. The
// last stage holds g~ and A~ back for the algebraic enforcement.
template <int MODE>
struct StageSink {
  const GridView &g;
  long long i;
  const StageArgs &a;
  double ug[6], uA[6];
  __device__ __forceinline__ void operator()(int v, double k) {
    const long long o = v * g.S + i;
    if (MODE < 0) {
      st_st(a.out + o, k);
      return;
    }
    double acc = MODE == 0 ? 0.0 : st_ld(a.acc + o);
    const double un = rk_combine<(MODE < 0 ? 0 : MODE), double>(st_ld(a.U + o), acc, k, a.dt);
    if (MODE < 3) st_st(a.acc + o, acc);
    if (!CCZ4_ENFORCE_RELOAD && MODE == 3 && v >= GXX && v <= GZZ) {
      ug[v - GXX] = un;
      return;
    }
    if (!CCZ4_ENFORCE_RELOAD && MODE == 3 && v >= AXX && v <= AZZ) {
      uA[v - AXX] = un;
      return;
    }
    st_st(a.out + o, un);
  }
  __device__ __forceinline__ void finish() {
    if (MODE != 3) return;
    if (CCZ4_ENFORCE_RELOAD) {
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        ug[c] = st_ld(a.out + (GXX + c) * g.S + i);
        uA[c] = st_ld(a.out + (AXX + c) * g.S + i);
      }
    }
    enforce_point<double>(ug, uA);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      st_st(a.out + (GXX + c) * g.S + i, ug[c]);
      st_st(a.out + (AXX + c) * g.S + i, uA[c]);
    }
  }
};

// Resident blocks of 128 threads per SM that a launch shape asks of the
// stage kernel: the default of the precision, one more (shape 1) or one
// fewer (shape 2).
template <class R, int SHAPE>
struct StageBlocks {
  static constexpr int base = std::is_same<R, float>::value ? CCZ4_INTERIOR_MIN_BLOCKS_MIXED : CCZ4_INTERIOR_MIN_BLOCKS;
  static constexpr int value = SHAPE == 1 ? base + 1 : SHAPE == 2 ? (base > 1 ? base - 1 : 1) : base;
};

// One interior point of the stage, its sums at place q of the derivative buffer.
template <int MODE, class R, bool MESH>
__device__ __forceinline__ void stage_point(const GridView &g, const Phys<R> &P, const LevelCoef<R> &LC,
                                            const StageBufs &b, const StageArgs &a, long long i, long long q) {
  constexpr bool MIXED = std::is_same<R, float>::value;
  // the patch (32-bit division: every state index is below 2^31) only where its level matters;
  // a run-time index into the parameter array makes ptxas keep a local copy of the array
  const int lev = MESH ? patch_level(g, (int)i / (g.p * g.p * g.p)) : 0;
  const StencilCoef<double> C = MESH ? LC.C[lev] : LC.C[0];
  const StencilCoef<R> CR = MESH ? LC.CR[lev] : LC.CR[0];
  const DerView<MIXED> N = der_view<MIXED>(g, b.der, b.mix, b.in, i, q);
  StageSink<MODE> sink{g, i, a};
  ccz4_rhs_point<double, R>(P, N, C, CR, sink);
  sink.finish();
}

// One thread per (evolved Sommerfeld ghost cell, field): the ghost-cell
// ODE (Eq. exa_sommerfeld_inter) with the cell's static geometry from
// g.ghost_geo, and the same stage update, no enforcement, FP64.
template <int MODE>
__device__ __forceinline__ void ghost_point(const GridView &g, const ccz4_params &P, const double *__restrict__ in,
                                            const double *__restrict__ ini, const StageArgs &a, long long id,
                                            int v) {
  const GhostGeo *gg = g.ghost_geo + id;
  const long long sn = __ldg(&gg->sn);
  if (sn < 0) return;
  const double geo = __ldg(&gg->geo), ir = __ldg(&gg->ir);
  // the field's speed, selected with static indices (a run-time index into
  // the parameter array would copy it to local memory)
  double cv = P.somm_speed[0];
#pragma unroll
  for (int q = 1; q < NV; ++q)
    if (q == v) cv = P.somm_speed[q];
  const long long o = v * g.S + g.n_points + id;
  const double qg = __ldg(in + o);
  const double qn = __ldg(in + v * g.S + sn);
  const double k = -cv * geo * (qg - qn) - cv * ir * (qg - __ldg(ini + o));
  if (MODE < 0) {
    a.out[o] = k;
    return;
  }
  double acc = MODE == 0 ? 0.0 : a.acc[o];
  const double un = rk_combine<(MODE < 0 ? 0 : MODE), double>(a.U[o], acc, k, a.dt);
  if (MODE < 3) a.acc[o] = acc;
  a.out[o] = un;
}

// All fields of one ghost cell: its geometry is read once and the 25 fields'
// loads are independent (consecutive cells, coalesced).
template <int MODE>
__device__ __forceinline__ void ghost_cell(const GridView &g, const ccz4_params &P, const StageBufs &b,
                                           const StageArgs &a, long long id) {
#pragma unroll 5
  for (int v = 0; v < NV; ++v) ghost_point<MODE>(g, P, b.in, b.ini, a, id, v);
}

// Next item of a warp from the device queue (g.queue).
__device__ __forceinline__ long long next_item(const GridView &g, int lane) {
  unsigned long long q = 0;
  if (lane == 0) q = atomicAdd(g.queue, 1ULL);
  return (long long)__shfl_sync(0xffffffffu, q, 0);
}

// First point of the window and the number of its points.
__device__ __forceinline__ long long window_begin(const GridView &g) { return (long long)g.w0 * (g.p * g.p * g.p); }
__device__ __forceinline__ long long window_points(const GridView &g) { return (long long)g.wn * (g.p * g.p * g.p); }

// Every interior point of the window, of every level, and with the first
// window every ghost cell.
// Flat launch (QUEUE false): the first ghost_blocks blocks take the ghost
// cells, the others one interior point per thread.
// Queue launch (QUEUE, the grid sized to the resident blocks): each warp
// takes items of 32 ghost cells or 32 interior points from the device counter
// g.queue until none is left; nothing waits on another thread.
template <int MODE, class R, bool MESH, bool QUEUE, int SHAPE = 0>
__global__ void __launch_bounds__(128, (StageBlocks<R, SHAPE>::value))
    algebra_kernel(GridView g, Phys<R> P, LevelCoef<R> LC, ccz4_params Pg, StageBufs b, StageArgs a, int ghost_blocks) {
  if (!QUEUE) {
    if ((int)blockIdx.x < ghost_blocks) {
      const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
      if (id < g.n_ghost) ghost_cell<MODE>(g, Pg, b, a, id);
      return;
    }
    const long long q = (long long)(blockIdx.x - ghost_blocks) * blockDim.x + threadIdx.x;
    if (q < window_points(g)) stage_point<MODE, R, MESH>(g, P, LC, b, a, window_begin(g) + q, q);
    return;
  }
  const int lane = threadIdx.x & 31;
  const long long gi = g.w0 == 0 ? (g.n_ghost + 31) / 32 : 0;  // items of ghost cells
  for (long long item = next_item(g, lane); (item - gi) * 32 < window_points(g); item = next_item(g, lane)) {
    if (item < gi) {
      const long long id = item * 32 + lane;
      if (id < g.n_ghost) ghost_cell<MODE>(g, Pg, b, a, id);
    } else {
      const long long q = (item - gi) * 32 + lane;
      if (q < window_points(g)) stage_point<MODE, R, MESH>(g, P, LC, b, a, window_begin(g) + q, q);
    }
  }
}

// Points of the window, and the ghost cells that go with it.
inline long long launch_points(const GridView &g) { return (long long)g.wn * g.p * g.p * g.p; }
inline long long launch_ghosts(const GridView &g) { return g.w0 == 0 ? g.n_ghost : 0; }

StencilCoef<double> coefs(double dx, const ccz4_params &P) {
  StencilCoef<double> C;
  C.c1 = 1.0 / (12.0 * dx);
  C.c2 = 1.0 / (12.0 * dx * dx);
  C.c3 = 1.0 / (144.0 * dx * dx);
  C.cko = P.ko_eps / (64.0 * dx);
  return C;
}

template <class R>
LevelCoef<R> level_coefs(const GridView &g, const ccz4_params &P) {
  LevelCoef<R> LC;
  for (int l = 0; l < MAX_LEVELS; ++l) {
    const StencilCoef<double> C = coefs(g.ldx[l], P);
    LC.C[l] = C;
    LC.CR[l] = StencilCoef<R>{R(C.c1), R(C.c2), R(C.c3), R(C.cko)};
  }
  return LC;
}

// Blocks of a queue launch: every SM filled with as many blocks as fit.
template <int MODE, class R, bool MESH>
long long queue_blocks() {
  int dev = 0, sms = 0, occ = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, algebra_kernel<MODE, R, MESH, true>, 128, 0);
  return (long long)sms * occ;
}

// Threads of a block: 128, or on a small grid one warp, so that the points
// spread over the SMs in shares of 32 (the FP64 pipe of the fullest SM sets
// the time: 27^3 points are 154 blocks of 128, two of them on some SM).
inline int stage_threads(long long points, int sms) { return points < 16LL * sms * 128 ? 32 : 128; }

template <int MODE, class R, bool MESH, int SHAPE>
cudaError_t launch_flat(const GridView &g, const ccz4_params &P, const StageBufs &b, const StageArgs &a,
                        cudaStream_t s) {
  const int t = stage_threads(launch_points(g), g.sms);
  const long long gb = (launch_ghosts(g) + t - 1) / t, nb = (launch_points(g) + t - 1) / t;
  if (gb + nb == 0) return cudaSuccess;
  algebra_kernel<MODE, R, MESH, false, SHAPE><<<(unsigned)(gb + nb), t, 0, s>>>(g, make_phys<R>(P), level_coefs<R>(g, P),
                                                                                P, b, a, (int)gb);
  return cudaGetLastError();
}

template <int MODE, class R, bool MESH>
cudaError_t launch_mode(const GridView &g, const ccz4_params &P, const StageBufs &b, const StageArgs &a,
                        cudaStream_t s) {
  if (g.queue) {
    const long long items = (launch_points(g) + 31) / 32 + (launch_ghosts(g) + 31) / 32, qb = queue_blocks<MODE, R, MESH>();
    if (qb <= 0) return cudaErrorInvalidConfiguration;
    if (items == 0) return cudaSuccess;
    const long long blocks = qb < (items + 3) / 4 ? qb : (items + 3) / 4;
    cudaError_t e = cudaMemsetAsync(g.queue, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    algebra_kernel<MODE, R, MESH, true><<<(unsigned)blocks, 128, 0, s>>>(g, make_phys<R>(P), level_coefs<R>(g, P), P, b,
                                                                         a, 0);
    return cudaGetLastError();
  }
  if (MODE >= 0 && (g.stage_shape == 1 || g.stage_shape == 2))
    return MESH ? launch_shaped_mesh(g, MODE, P, b, a, s) : launch_shaped_uniform(g, MODE, P, b, a, s);
  return launch_flat<MODE, R, MESH, 0>(g, P, b, a, s);
}

template <int MODE, bool MESH>
cudaError_t launch_prec(const GridView &g, const ccz4_params &P, const StageBufs &b, const StageArgs &a,
                        cudaStream_t s) {
  if (P.precision == CCZ4_PREC_MIXED) return launch_mode<MODE, float, MESH>(g, P, b, a, s);
  return launch_mode<MODE, double, MESH>(g, P, b, a, s);
}

// stage -1: plain right-hand side; 0..3: RK4 stage
template <bool MESH>
cudaError_t launch_stage(const GridView &g, const ccz4_params &P, int stage, const StageBufs &b, const StageArgs &a,
                         cudaStream_t s) {
  switch (stage) {
    case -1: return launch_prec<-1, MESH>(g, P, b, a, s);
    case 0: return launch_prec<0, MESH>(g, P, b, a, s);
    case 1: return launch_prec<1, MESH>(g, P, b, a, s);
    case 2: return launch_prec<2, MESH>(g, P, b, a, s);
    case 3: return launch_prec<3, MESH>(g, P, b, a, s);
    default: return cudaErrorInvalidValue;
  }
}

template <class R, bool MESH, int SHAPE>
cudaError_t launch_shape_of(const GridView &g, int stage, const ccz4_params &P, const StageBufs &b, const StageArgs &a,
                            cudaStream_t s) {
  switch (stage) {
    case 0: return launch_flat<0, R, MESH, SHAPE>(g, P, b, a, s);
    case 1: return launch_flat<1, R, MESH, SHAPE>(g, P, b, a, s);
    case 2: return launch_flat<2, R, MESH, SHAPE>(g, P, b, a, s);
    case 3: return launch_flat<3, R, MESH, SHAPE>(g, P, b, a, s);
    default: return cudaErrorInvalidValue;
  }
}

template <bool MESH>
cudaError_t launch_shaped(const GridView &g, int stage, const ccz4_params &P, const StageBufs &b, const StageArgs &a,
                          cudaStream_t s) {
  if (P.precision == CCZ4_PREC_MIXED)
    return g.stage_shape == 1 ? launch_shape_of<float, MESH, 1>(g, stage, P, b, a, s)
                              : launch_shape_of<float, MESH, 2>(g, stage, P, b, a, s);
  return g.stage_shape == 1 ? launch_shape_of<double, MESH, 1>(g, stage, P, b, a, s)
                            : launch_shape_of<double, MESH, 2>(g, stage, P, b, a, s);
}

}  // namespace
}  // namespace ccz4
