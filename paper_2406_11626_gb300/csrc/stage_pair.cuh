// One launch per FP64 RK stage of a large grid: a block's warps split into two
// parts that run side by side, one patch apart.
//
// The derivative pass waits on memory, shared memory and integer units and
// needs little of the FP64 pipe; the algebra keeps that pipe busy and issues
// in 9 % of the cycles. As two launches they run one after the other (ncu: the
// pipe 91 % busy in the second, 30 % in the first). Here one part of a block's
// threads takes the derivatives of its next patch while the other
// evaluates the points of the one before. The parts meet at a barrier per
// patch; nothing waits on another block, and a block reads no derivatives but
// its own: it keeps those of two patches, in places of its own of the derivative
// buffer. Streams do not do it: the same overlap by two streams and chunks
// of patches took 37.8 ms (4 chunks) and 46.0 ms (16) as a graph, the blocks of
// one kernel filling the SMs before the other's.
//
// The registers are split by setmaxnreg. One RK4 step at 144^3 as two launches
// 36.2 ms; threads of the two parts and their registers 256 + 384 (56, 120)
// 39.0, 384 + 256 (56, 152) 32.8, 512 + 256 (48, 144) 32.6, 512 + 384 (40, 112)
// 31.7, two blocks of 256 + 128 (56, 128) 33.3, 384 + 384 (48, 112) 31.6: the
// algebra wants 12 warps to cover its latency, the derivatives 12 to keep up. With
// their conversions to FP64 in integers (CVT false) 30.4; with an algebra of 100
// operations less 28.5; with no FP64 operation of theirs issued in vain 26.46, and
// 26.27 with (40, 120), 26.5 with (56, 104), 38.8 with 256 + 384 (56, 120). On a mesh
// the derivatives are the longer part (interpolated halo points): two levels of 2240
// patches 18.9 ms with 384 + 384, 18.7 with 512 + 384, 17.7 with 512 + 256 (48, 144),
// 17.8 with 640 + 256; of late 16.7, and (40, 160) 16.8, (56, 128) 17.1, 384 + 384 (48,
// 112) 17.5. What bounds it: the FP64 pipe (1187
// operations a point, 22.5 of the 26.2 ms) and the stalls that the algebra's warps
// leave open.
//
// Mixed precision keeps two launches: there the derivative pass is the longer
// part and wants the whole SM (15.0 ms against 15.2 at best).
#pragma once

// the derivatives are read back in the launch that writes them: coherent loads through L2
#define CCZ4_DER_LOAD __ldcg
#include "derive_edge.cuh"
#include "stage_kernels.cuh"

namespace ccz4 {

cudaError_t prepare_pair_uniform();
cudaError_t prepare_pair_mesh();
cudaError_t launch_pair_uniform(const GridView &g, const ccz4_params &P, int stage, double *tile, double *mix, double *der,
                                const double *in, const double *ini, const StageArgs &a, cudaStream_t s);
cudaError_t launch_pair_mesh(const GridView &g, const ccz4_params &P, int stage, double *tile, double *mix, double *der,
                             const double *in, const double *ini, const StageArgs &a, cudaStream_t s);

namespace {

// The place that block `block` of `blocks` gives the derivatives of patch n: one of two, which take turns.
// A patch's are overwritten two rounds later, when the barrier of the round between has shown them read.
__device__ __forceinline__ int pair_place(int n, int block, int blocks) { return block + (n / blocks % 2) * blocks; }

template <bool MESH>
struct Split {
  // threads of the derivatives and of the algebra, and the registers each of them gets
  static constexpr int derive = MESH ? 512 : 384, algebra = MESH ? 256 : 384, threads = derive + algebra;
  static constexpr int derive_regs = MESH ? 48 : 40, algebra_regs = MESH ? 144 : 120;
  // Registers a thread of the launch (what 65536 leave for its threads, in steps
  // of 8). The parts may not ask for more in sum: they would wait for ever.
  static constexpr int regs = 65536 / threads / 8 * 8;
  static_assert(derive * derive_regs + algebra * algebra_regs <= threads * regs, "registers");
  static_assert(derive % 128 == 0 && algebra % 128 == 0, "whole warpgroups");
};

template <int MODE, bool MESH, int PF>
__global__ void __launch_bounds__(Split<MESH>::threads, 1)
    pair_kernel(GridView g, Phys<double> P, LevelCoef<double> LC, LevelScale ls, ccz4_params Pg, FieldList fl,
                double *tile, double *mix, double *der, const double *__restrict__ in, const double *__restrict__ ini,
                StageArgs a) {
  extern __shared__ double smem[];
  using X = Split<MESH>;
  constexpr int P3 = PF * PF * PF;
  if (threadIdx.x < X::derive) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(X::derive_regs));
#pragma unroll 1
    for (int n = blockIdx.x; n < g.n_patches; n += gridDim.x) {
      derive_edge<MESH ? FROM_MESH : FROM_LEVEL, X::derive, PF, false>(g, in, tile, mix, der, ls, fl, n,
                                                                       pair_place(n, blockIdx.x, gridDim.x), 0, 1, smem,
                                                                       threadIdx.x, 1);
      block_sync<X::threads>(2);
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(X::algebra_regs));
    const StageBufs b{der, mix, in, ini};
    const int tid = threadIdx.x - X::derive;
    // the ghost cells while the first patch's derivatives are taken
#pragma unroll 1
    for (long long id = (long long)blockIdx.x * X::algebra + tid; id < g.n_ghost;
         id += (long long)gridDim.x * X::algebra)
      ghost_cell<MODE>(g, Pg, b, a, id);
#pragma unroll 1
    for (int n = blockIdx.x; n < g.n_patches; n += gridDim.x) {
      block_sync<X::threads>(2);  // patch n's derivatives are written
#pragma unroll 1
      for (int q = tid; q < P3; q += X::algebra)
        stage_point<MODE, double, MESH>(g, P, LC, b, a, (long long)n * P3 + q,
                                        (long long)pair_place(n, blockIdx.x, gridDim.x) * P3 + q);
    }
  }
}

template <int MODE, bool MESH, int PF>
cudaError_t prepare_pair_one() {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, pair_kernel<MODE, MESH, PF>);
  if (e != cudaSuccess) return e;
  if (fa.numRegs != Split<MESH>::regs) return cudaErrorInvalidConfiguration;  // the split above would not add up
  return cudaFuncSetAttribute(pair_kernel<MODE, MESH, PF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)edge_smem_bytes(PF));
}

template <int MODE, bool MESH, int PF>
cudaError_t launch_pair_one(const GridView &g, const ccz4_params &P, double *tile, double *mix, double *der,
                            const double *in, const double *ini, const StageArgs &a, cudaStream_t s) {
  pair_kernel<MODE, MESH, PF><<<g.n_patches < g.sms ? g.n_patches : g.sms, Split<MESH>::threads, edge_smem_bytes(PF), s>>>(
      g, make_phys<double>(P), level_coefs<double>(g, P), level_scale(g), P, all_fields(), tile, mix, der, in, ini, a);
  return cudaGetLastError();
}

template <bool MESH, int PF>
cudaError_t prepare_pair_as() {
  cudaError_t e = prepare_pair_one<0, MESH, PF>();
  if (e == cudaSuccess) e = prepare_pair_one<1, MESH, PF>();
  if (e == cudaSuccess) e = prepare_pair_one<2, MESH, PF>();
  if (e == cudaSuccess) e = prepare_pair_one<3, MESH, PF>();
  return e;
}

template <bool MESH, int PF>
cudaError_t launch_pair_as(const GridView &g, const ccz4_params &P, int stage, double *tile, double *mix, double *der,
                           const double *in, const double *ini, const StageArgs &a, cudaStream_t s) {
  switch (stage) {
    case 0: return launch_pair_one<0, MESH, PF>(g, P, tile, mix, der, in, ini, a, s);
    case 1: return launch_pair_one<1, MESH, PF>(g, P, tile, mix, der, in, ini, a, s);
    case 2: return launch_pair_one<2, MESH, PF>(g, P, tile, mix, der, in, ini, a, s);
    case 3: return launch_pair_one<3, MESH, PF>(g, P, tile, mix, der, in, ini, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace
}  // namespace ccz4
