// mixed-precision (GLEMUR_MIXED: FP32 storage and stencils, float-float determinants, FP64 reductions) instantiations of the mimetic-current stage kernels.
#include "stage_march.cuh"

namespace glemur {

// 8 warps (tiles of 64 x 8 nodes), 2 CTAs per SM.  `maps` null: the loader
// without TMA.
cudaError_t launch_f32_mimetic(const StageArgs<float>& a, const TmaMaps* maps, int stage,
                               dim3 grid, cudaStream_t s) {
  return launch_stage_march_t<8, 2>(a, maps, stage, grid, s);
}

cudaError_t prepare_f32_mimetic() { return prepare_stage_march_t<8, 2>(); }

int ctas_per_sm_f32_mimetic(bool tma) { return stage_march_ctas_per_sm_t<8, 2>(tma); }

// Tile extents (nodes); the stage-input box is 4 rows higher, the B0 box 2,
// both 8 columns wider.
int tile_cols_f32_mimetic() { return MX; }
int tile_rows_f32_mimetic() { return MarchGeo<8>::TH; }

}  // namespace glemur
