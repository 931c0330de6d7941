// One launch per RK stage (CCZ4_LAUNCH_FUSED): a cooperative kernel whose
// blocks first take the derivatives of all patches (one patch per block at
// a time, the pass of derive.cuh), wait for one another at a grid-wide barrier,
// then evolve the Sommerfeld ghost cells and the interior points (items of 32
// per warp, strided over the grid); on a grid with more patches than its
// derivative buffer holds, window after window, with a barrier between. This is
// the paper's enclave batching taken to a whole stage: every patch of every level
// in one task.
// Compiled for 9^3 patches (the derivative pass's instance for that edge) and
// the RK stages; the restriction after a step stays its own launch.
//
// The derivatives are written by the first phase of the same launch, so they
// are read back with coherent loads through L2; the grid barrier orders them.
#define CCZ4_DER_LOAD __ldcg
#include <cooperative_groups.h>

#include "derive_edge.cuh"
#include "stage_kernels.cuh"

namespace ccz4 {
namespace {

constexpr int FUSED_THREADS = 128;
constexpr int FUSED_PF = 9;

template <int MODE, class R, bool MESH>
__global__ void __launch_bounds__(FUSED_THREADS, (StageBlocks<R, 0>::value))
    fused_stage_kernel(GridView g, Phys<R> P, LevelCoef<R> LC, LevelScale ls, ccz4_params Pg, FieldList fl,
                       double *tile, double *mix, double *der, const double *__restrict__ in,
                       const double *__restrict__ ini, StageArgs a) {
  extern __shared__ double smem[];
  const StageBufs b{der, mix, in, ini};
  const int lane = threadIdx.x & 31;
  const long long warps = (long long)gridDim.x * (FUSED_THREADS / 32);
  constexpr int P3 = FUSED_PF * FUSED_PF * FUSED_PF;
#pragma unroll 1
  for (int w0 = 0; w0 < g.n_patches; w0 += g.wcap) {  // (the derivative buffer holds wcap patches)
    const int wn = g.n_patches - w0 < g.wcap ? g.n_patches - w0 : g.wcap;
    if (w0 > 0) cooperative_groups::this_grid().sync();  // the sums of the window before are read
    for (int k = blockIdx.x; k < wn; k += gridDim.x) {
      constexpr int SRC = MESH ? FROM_MESH : FROM_LEVEL;
      const int n = w0 + k;
      if constexpr (std::is_same<R, float>::value)
        derive_patch<SRC, true, FUSED_THREADS, FUSED_PF, NV>(g, in, tile, mix, der, ls, fl, n, k, 0, 1, false, smem);
      else
        derive_edge<SRC, FUSED_THREADS, FUSED_PF, true>(g, in, tile, mix, der, ls, fl, n, k, 0, 1, smem, threadIdx.x, 0);
      __syncthreads();  // the next patch's source table overwrites this one's shared memory
    }
    cooperative_groups::this_grid().sync();
    const long long gi = w0 == 0 ? (g.n_ghost + 31) / 32 : 0, points = (long long)wn * P3;
    for (long long item = (long long)blockIdx.x * (FUSED_THREADS / 32) + threadIdx.x / 32; (item - gi) * 32 < points;
         item += warps) {
      if (item < gi) {
        const long long id = item * 32 + lane;
        if (id < g.n_ghost) ghost_cell<MODE>(g, Pg, b, a, id);
      } else {
        const long long q = (item - gi) * 32 + lane;
        if (q < points) stage_point<MODE, R, MESH>(g, P, LC, b, a, (long long)w0 * P3 + q, q);
      }
    }
  }
}

template <class R>
size_t fused_smem_bytes() {
  return std::is_same<R, float>::value ? derive_smem_bytes(FUSED_PF) : edge_smem_bytes(FUSED_PF);
}

template <int MODE, class R, bool MESH>
const void *fused_fn() {
  return (const void *)fused_stage_kernel<MODE, R, MESH>;
}

// Every instance, for the shared-memory attribute and the occupancy query.
const void *fused_any(int mode, bool mixed, bool mesh) {
#define CCZ4_FUSED_CASE(M)                                                                       \
  case M:                                                                                        \
    return mixed ? (mesh ? fused_fn<M, float, true>() : fused_fn<M, float, false>())             \
                 : (mesh ? fused_fn<M, double, true>() : fused_fn<M, double, false>());
  switch (mode) {
    CCZ4_FUSED_CASE(0)
    CCZ4_FUSED_CASE(1)
    CCZ4_FUSED_CASE(2)
    CCZ4_FUSED_CASE(3)
  }
#undef CCZ4_FUSED_CASE
  return nullptr;
}

template <int MODE, class R, bool MESH>
cudaError_t launch_fused_as(const GridView &g, const ccz4_params &P, double *tile, double *mix, double *der,
                            const double *in, const double *ini, const StageArgs &a, cudaStream_t s) {
  const void *fn = fused_fn<MODE, R, MESH>();
  const size_t smem = fused_smem_bytes<R>();
  int dev = 0, sms = 0, occ = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, FUSED_THREADS, smem);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaErrorInvalidConfiguration;
  LevelCoef<R> LC = level_coefs<R>(g, P);
  FieldList fl = all_fields();
  GridView gv = g;
  Phys<R> ph = make_phys<R>(P);
  LevelScale ls = level_scale(g);
  ccz4_params Pg = P;
  StageArgs av = a;
  void *args[] = {&gv, &ph, &LC, &ls, &Pg, &fl, &tile, &mix, &der, (void *)&in, (void *)&ini, &av};
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // all blocks resident: the grid barrier may wait for every one
  attr[0].val.cooperative = 1;
  cfg.gridDim = dim3((unsigned)(sms * occ));
  cfg.blockDim = dim3(FUSED_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

template <int MODE>
cudaError_t launch_fused_mode(const GridView &g, const ccz4_params &P, double *tile, double *mix, double *der,
                              const double *in, const double *ini, const StageArgs &a, cudaStream_t s) {
  const bool mixed = P.precision == CCZ4_PREC_MIXED, mesh = g.src != nullptr;
  if (mixed)
    return mesh ? launch_fused_as<MODE, float, true>(g, P, tile, mix, der, in, ini, a, s)
                : launch_fused_as<MODE, float, false>(g, P, tile, mix, der, in, ini, a, s);
  return mesh ? launch_fused_as<MODE, double, true>(g, P, tile, mix, der, in, ini, a, s)
              : launch_fused_as<MODE, double, false>(g, P, tile, mix, der, in, ini, a, s);
}

}  // namespace

cudaError_t prepare_fused() {
  for (int m = 0; m < 4; ++m)
    for (int x = 0; x < 2; ++x)
      for (int h = 0; h < 2; ++h) {
        const int bytes = (int)(x ? fused_smem_bytes<float>() : fused_smem_bytes<double>());
        cudaError_t e = cudaFuncSetAttribute(fused_any(m, x, h), cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
      }
  return cudaSuccess;
}

cudaError_t launch_fused_stage(const GridView &g, const ccz4_params &P, int stage, double dt, double *tile,
                               double *mix, double *der, const double *in, const double *ini, const double *U,
                               double *acc, double *out, cudaStream_t s) {
  if (g.p != FUSED_PF || stage < 0 || stage > 3) return cudaErrorInvalidValue;
  const StageArgs a{U, acc, out, dt};
  switch (stage) {
    case 0: return launch_fused_mode<0>(g, P, tile, mix, der, in, ini, a, s);
    case 1: return launch_fused_mode<1>(g, P, tile, mix, der, in, ini, a, s);
    case 2: return launch_fused_mode<2>(g, P, tile, mix, der, in, ini, a, s);
    default: return launch_fused_mode<3>(g, P, tile, mix, der, in, ini, a, s);
  }
}

}  // namespace ccz4
