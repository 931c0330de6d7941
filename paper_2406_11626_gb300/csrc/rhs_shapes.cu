// Algebra kernels of a single level in the launch shapes other than the default
// (one resident block more or fewer per SM), for the autotuner; a translation
// unit of their own so they compile in parallel.
#include "stage_kernels.cuh"

namespace ccz4 {

cudaError_t launch_shaped_uniform(const GridView &g, int stage, const ccz4_params &P, const StageBufs &b,
                             const StageArgs &a, cudaStream_t s) {
  return launch_shaped<false>(g, stage, P, b, a, s);
}

}  // namespace ccz4
