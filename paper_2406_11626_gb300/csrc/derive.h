// Layout of the derivative buffer and the launches of the derivative pass
// (derive.cuh has the kernels' bodies, derive.cu the kernels).
#pragma once

#include "ccz4_internal.cuh"

namespace ccz4 {

// ---- layout of the derivative buffer ------------------------------------------------
// Slots of one value for each point of the buffer's patches (GridView::wcap; the
// points of the pass's window in order), point index fastest. FP64 (and the
// first-order formulation): 4 v + k for the first-derivative sum along k and
// 4 v + 3 for the dissipation sum of field v; from 4 NV on, three pure second
// sums for each field of the mixed-derivative buffer, in its order.
// Mixed precision: alpha and phi hold 7 FP64 slots each (first, dissipation,
// pure), then the other fields FP32 slots in the same order as FP64 ones.
constexpr int DER_SLOTS = 4 * NV + 33;
__host__ __device__ __forceinline__ constexpr int der_second(int v) { return mix_slot(v) < 0 ? -1 : mix_slot(v) / 3; }
// mixed precision: position of an FP32 field among the FP32 fields, and among those with second derivatives
__host__ __device__ __forceinline__ constexpr int der_f(int v) { return v < ALPHA ? v : v < PHI ? v - 1 : v - 2; }
__host__ __device__ __forceinline__ constexpr int der_f2(int v) { return v < ALPHA ? v : v - 1; }
constexpr int DER_D = 14;        // FP64 slots of the mixed precision
constexpr int DER_F = 4 * 23;    // FP32 slots before the pure second sums
__host__ __device__ __forceinline__ constexpr bool der_f32(bool mixed, int v) { return mixed && v != ALPHA && v != PHI; }

// Fields that a derivative pass takes; FIELD_NO_SUMS marks one of which only
// the tile and the mixed derivatives are wanted.
constexpr int FIELD_NO_SUMS = 0x80;
struct FieldList {
  unsigned char f[64];
  int n;
};

// Launches (derive.cu). The tile sources are those of the grid (a level or a
// mesh) or, from_tile, the tile buffer as ccz4_fill_halos or, mixed,
// ccz4_fill_halos_for wrote it (mix is left as it is).
cudaError_t launch_derive(const GridView &g, const double *src, double *tile, double *mix, double *der,
                          const FieldList &fl, bool mixed, bool from_tile, bool tile_out, cudaStream_t s);
cudaError_t launch_derive_fo(const GridView &g, const double *src, double *der, const FieldList &fl, cudaStream_t s);
cudaError_t prepare_derive();  // shared-memory limits; once per grid, outside any stream capture
// The 25 fields in the order the pass takes them: those with second derivatives first, so that the
// groups of a small grid share them out evenly.
FieldList all_fields();

}  // namespace ccz4
