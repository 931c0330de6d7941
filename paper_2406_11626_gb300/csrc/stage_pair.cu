// The one-launch stages (stage_pair.cuh) of a single level.
#include "stage_pair.cuh"

namespace ccz4 {

cudaError_t prepare_pair_uniform() { return prepare_pair_as<false, 9>(); }

cudaError_t launch_pair_uniform(const GridView &g, const ccz4_params &P, int stage, double *tile, double *mix, double *der,
                         const double *in, const double *ini, const StageArgs &a, cudaStream_t s) {
  return launch_pair_as<false, 9>(g, P, stage, tile, mix, der, in, ini, a, s);
}

cudaError_t prepare_pair(bool mesh) { return mesh ? prepare_pair_mesh() : prepare_pair_uniform(); }

cudaError_t launch_pair_stage(const GridView &g, const ccz4_params &P, int stage, double dt, double *tile, double *mix,
                              double *der, const double *in, const double *ini, const double *U, double *acc, double *out,
                              cudaStream_t s) {
  const StageArgs a{U, acc, out, dt};
  return g.src ? launch_pair_mesh(g, P, stage, tile, mix, der, in, ini, a, s)
               : launch_pair_uniform(g, P, stage, tile, mix, der, in, ini, a, s);
}

}  // namespace ccz4
