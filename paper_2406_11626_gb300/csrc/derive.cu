// The derivative pass (derive.cuh): kernels and launches.
#include "derive_edge.cuh"

namespace ccz4 {
namespace {

template <int SRC, bool MIXED, int SHAPE, int PF, int NF>
__global__ void __launch_bounds__(FILL_SHAPE_THREADS[SHAPE], (PF == 9 ? 1024 : 768) / FILL_SHAPE_THREADS[SHAPE])
    derive_kernel(GridView g, const double *__restrict__ src, double *tile, double *__restrict__ mix,
                  double *__restrict__ der, LevelScale ls, FieldList fl, bool tile_out) {
  extern __shared__ double smem[];
  derive_patch<SRC, MIXED, FILL_SHAPE_THREADS[SHAPE], PF, NF>(g, src, tile, mix, der, ls, fl, g.w0 + blockIdx.x, blockIdx.x,
                                                              blockIdx.y, gridDim.y, tile_out, smem);
}

template <int SRC, int PF>
__global__ void __launch_bounds__(EdgeShape<PF>::threads, EdgeShape<PF>::blocks)
    derive_edge_kernel(GridView g, const double *__restrict__ src, double *tile, double *__restrict__ mix,
                       double *__restrict__ der, LevelScale ls, FieldList fl) {
  extern __shared__ double smem[];
  derive_edge<SRC, EdgeShape<PF>::threads, PF, true>(g, src, tile, mix, der, ls, fl, g.w0 + blockIdx.x, blockIdx.x,
                                                     blockIdx.y, gridDim.y, smem, threadIdx.x, 0);
}

// One field per block, 9^3 patches: small grids. Four blocks of 54 KB fit an SM, so 24 patches are one wave of
// 600 blocks (27 are 675, a wave and a tenth).
constexpr int ONE_THREADS = 256;
template <int SRC>
__global__ void __launch_bounds__(ONE_THREADS, 4)
    derive_field_kernel(GridView g, const double *__restrict__ src, double *tile, double *__restrict__ mix,
                        double *__restrict__ der, LevelScale ls, FieldList fl) {
  extern __shared__ double smem[];
  derive_edge<SRC, ONE_THREADS, 9, true, true>(g, src, tile, mix, der, ls, fl, g.w0 + blockIdx.x, blockIdx.x, blockIdx.y,
                                               fl.n, smem, threadIdx.x, 0);
}

// Field groups per patch. A block's set-up (the source table) is shared by
// the fields it takes, so a grid of many patches gives each block all fields;
// a grid of few patches splits them into about six blocks an SM, whatever number
// of them is resident (9^3: three or four, 12^3: one, so that 140 patches of 12^3
// in seven groups are 6.4 waves).
int field_groups(const GridView &g, const FieldList &fl) {
  const int want = 6 * g.sms;
  int k = g.wn > 0 ? (want + g.wn - 1) / g.wn : 1;
  k = k < 1 ? 1 : k;
  return k < fl.n ? k : fl.n;
}

template <int SRC, bool MIXED, int SHAPE, int PF, int NF>
cudaError_t launch_one(const GridView &g, const double *src, double *tile, double *mix, double *der,
                       const FieldList &fl, bool tile_out, cudaStream_t s) {
  const dim3 grid(g.wn, field_groups(g, fl));
  derive_kernel<SRC, MIXED, SHAPE, PF, NF><<<grid, FILL_SHAPE_THREADS[SHAPE], derive_smem_bytes(g.p), s>>>(
      g, src, tile, mix, der, level_scale(g), fl, tile_out);
  return cudaGetLastError();
}

template <int SRC, int PF>
cudaError_t launch_fixed(const GridView &g, const double *src, double *tile, double *mix, double *der,
                         const FieldList &fl, cudaStream_t s) {
  if (PF == 9 && field_groups(g, fl) == fl.n) {
    derive_field_kernel<SRC><<<dim3(g.wn, fl.n), ONE_THREADS, edge_smem_bytes(9, true), s>>>(
        g, src, tile, mix, der, level_scale(g), fl);
    return cudaGetLastError();
  }
  derive_edge_kernel<SRC, PF><<<dim3(g.wn, field_groups(g, fl)), EdgeShape<PF>::threads, edge_smem_bytes(PF), s>>>(
      g, src, tile, mix, der, level_scale(g), fl);
  return cudaGetLastError();
}

template <int SRC, bool MIXED, int SHAPE>
cudaError_t launch_edge(const GridView &g, const double *src, double *tile, double *mix, double *der,
                        const FieldList &fl, bool tile_out, cudaStream_t s) {
  if (g.p == 9) return launch_one<SRC, MIXED, SHAPE, 9, NV>(g, src, tile, mix, der, fl, tile_out, s);
  if constexpr (SHAPE == 0) {
    return launch_one<SRC, MIXED, 0, 0, NV>(g, src, tile, mix, der, fl, tile_out, s);
  } else {
    return launch_edge<SRC, MIXED, 0>(g, src, tile, mix, der, fl, tile_out, s);
  }
}

template <int SRC, bool MIXED>
cudaError_t launch_shape(const GridView &g, const double *src, double *tile, double *mix, double *der,
                         const FieldList &fl, bool tile_out, cudaStream_t s) {
  if constexpr (SRC != FROM_TILE && !MIXED) {
    // All 25 fields (a right-hand side): the edges of the study of patch sizes that leave room for the
    // widened first derivatives. The monitors' passes, which leave the FP64 pipe idle and write the
    // tiles too, stay with the general body (constraints at 144^3: 5.84 ms with it, 6.09 otherwise).
    if (!tile_out) {
      if (g.p == 9) return launch_fixed<SRC, 9>(g, src, tile, mix, der, fl, s);
      if (g.p == 12) return launch_fixed<SRC, 12>(g, src, tile, mix, der, fl, s);
      if (g.p == 6) return launch_fixed<SRC, 6>(g, src, tile, mix, der, fl, s);
    }
  } else if constexpr (SRC != FROM_TILE) {
    if (g.fill_shape == 1) return launch_edge<SRC, MIXED, 1>(g, src, tile, mix, der, fl, tile_out, s);
    if (g.fill_shape == 3) return launch_edge<SRC, MIXED, 3>(g, src, tile, mix, der, fl, tile_out, s);
  }
  return launch_edge<SRC, MIXED, 0>(g, src, tile, mix, der, fl, tile_out, s);
}

template <int SRC, bool MIXED, int SHAPE, int PF, int NF>
cudaError_t prepare_one(int p) {
  return cudaFuncSetAttribute(derive_kernel<SRC, MIXED, SHAPE, PF, NF>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, (int)derive_smem_bytes(p));
}

template <int SRC, int PF>
cudaError_t prepare_fixed() {
  return cudaFuncSetAttribute(derive_edge_kernel<SRC, PF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)edge_smem_bytes(PF));
}

template <int SRC, bool MIXED>
cudaError_t prepare_source() {
  cudaError_t e = prepare_one<SRC, MIXED, 0, 9, NV>(9);
  if constexpr (SRC != FROM_TILE && !MIXED) {
    if (e == cudaSuccess) e = prepare_fixed<SRC, 9>();
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(derive_field_kernel<SRC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)edge_smem_bytes(9, true));
    if (e == cudaSuccess) e = prepare_fixed<SRC, 12>();
    if (e == cudaSuccess) e = prepare_fixed<SRC, 6>();
  }
  if (e == cudaSuccess) e = prepare_one<SRC, MIXED, 0, 0, NV>(MAX_P);
  if constexpr (SRC != FROM_TILE && MIXED) {
    if (e == cudaSuccess) e = prepare_one<SRC, MIXED, 1, 9, NV>(9);
    if (e == cudaSuccess) e = prepare_one<SRC, MIXED, 3, 9, NV>(9);
  }
  return e;
}

}  // namespace

cudaError_t prepare_derive() {
  cudaError_t e = prepare_source<FROM_LEVEL, false>();
  if (e == cudaSuccess) e = prepare_source<FROM_LEVEL, true>();
  if (e == cudaSuccess) e = prepare_source<FROM_MESH, false>();
  if (e == cudaSuccess) e = prepare_source<FROM_MESH, true>();
  if (e == cudaSuccess) e = prepare_source<FROM_TILE, false>();
  if (e == cudaSuccess) e = prepare_source<FROM_TILE, true>();
  if (e == cudaSuccess) e = prepare_one<FROM_LEVEL, false, 0, 9, 58>(9);
  if (e == cudaSuccess) e = prepare_one<FROM_LEVEL, false, 0, 0, 58>(MAX_P);
  return e;
}

FieldList all_fields() {
  FieldList fl;
  fl.n = 0;
  for (int pass = 0; pass < 2; ++pass)
    for (int v = 0; v < NV; ++v)
      if ((mix_slot(v) >= 0) == (pass == 0)) fl.f[fl.n++] = (unsigned char)v;
  return fl;
}

cudaError_t launch_derive(const GridView &g, const double *src, double *tile, double *mix, double *der,
                          const FieldList &fl, bool mixed, bool from_tile, bool tile_out, cudaStream_t s) {
  if (g.wn == 0 || fl.n == 0) return cudaSuccess;
  if (from_tile)
    return mixed ? launch_shape<FROM_TILE, true>(g, src, tile, mix, der, fl, false, s)
                 : launch_shape<FROM_TILE, false>(g, src, tile, mix, der, fl, false, s);
  if (g.src)
    return mixed ? launch_shape<FROM_MESH, true>(g, src, tile, mix, der, fl, false, s)
                 : launch_shape<FROM_MESH, false>(g, src, tile, mix, der, fl, tile_out, s);
  return mixed ? launch_shape<FROM_LEVEL, true>(g, src, tile, mix, der, fl, false, s)
               : launch_shape<FROM_LEVEL, false>(g, src, tile, mix, der, fl, tile_out, s);
}

cudaError_t launch_derive_fo(const GridView &g, const double *src, double *der, const FieldList &fl, cudaStream_t s) {
  if (g.wn == 0 || fl.n == 0) return cudaSuccess;
  if (g.p == 9) return launch_one<FROM_LEVEL, false, 0, 9, 58>(g, src, nullptr, nullptr, der, fl, false, s);
  return launch_one<FROM_LEVEL, false, 0, 0, 58>(g, src, nullptr, nullptr, der, fl, false, s);
}

}  // namespace ccz4
