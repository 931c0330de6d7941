// Stage kernels of refined meshes: each thread takes the stencil
// coefficients of its patch's level.
#include "stage_kernels.cuh"

namespace ccz4 {

cudaError_t launch_stage_mesh(const GridView &g, const ccz4_params &P, int stage, const StageBufs &b,
                              const StageArgs &a, cudaStream_t s) {
  return launch_stage<true>(g, P, stage, b, a, s);
}

}  // namespace ccz4
