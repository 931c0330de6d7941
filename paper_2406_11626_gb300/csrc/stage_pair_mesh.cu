// The one-launch stages (stage_pair.cuh) of refined meshes.
#include "stage_pair.cuh"

namespace ccz4 {

cudaError_t prepare_pair_mesh() { return prepare_pair_as<true, 9>(); }

cudaError_t launch_pair_mesh(const GridView &g, const ccz4_params &P, int stage, double *tile, double *mix, double *der,
                         const double *in, const double *ini, const StageArgs &a, cudaStream_t s) {
  return launch_pair_as<true, 9>(g, P, stage, tile, mix, der, in, ini, a, s);
}

}  // namespace ccz4
