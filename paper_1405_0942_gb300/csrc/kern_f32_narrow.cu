// mixed-precision (GLEMUR_MIXED) mimetic-current stages on 32 x 8 tiles, one node per thread, for grids whose rows waste half of the march's last tile (choose_narrow).
#include "stage_kernels.cuh"

namespace glemur {

cudaError_t launch_f32_narrow(const StageArgs<float>& a, int stage, dim3 grid, cudaStream_t s) {
  return launch_stage_t<float, float, 0, 3>(a, stage, grid, s);
}

cudaError_t prepare_f32_narrow() { return prepare_stage_t<float, float, 0, 3>(); }

int ctas_per_sm_f32_narrow() { return stage_ctas_per_sm_t<float, float, 0, 3>(); }

}  // namespace glemur
