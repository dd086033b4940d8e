// fused_fp32_pair.cu -- binary32 stage kernels in which each thread owns two
// columns of a 64 x 8 tile (x and x + 32), computed together in f32x2
// (both accumulator kinds).  Shared-memory records hold both columns'
// values side by side, so every record access moves two points.
#include "fused_stage.cuh"

namespace sbli {

cudaError_t launch_fused_fp32_pair(const StageArgs& a, const Coef<float>& cf, const FusedConfig& cfg, bool in_fp64,
                                   bool df, bool rhs_only, cudaStream_t s) {
  if (cfg.ty != 8) return cudaErrorInvalidValue;
  const Coef<f32x2> c = both_lanes(cf);
  if (rhs_only) {
    if (in_fp64) return launch_fused_t<f32x2, double, float, 8, true, false>(a, c, s);
    return launch_fused_t<f32x2, float, float, 8, true, false>(a, c, s);
  }
  if (df) {
    if (a.ke_partials) return launch_fused_t<f32x2, float, float, 8, false, true, true>(a, c, s);
    return launch_fused_t<f32x2, float, float, 8, false, false, true>(a, c, s);
  }
  if (in_fp64) return cudaErrorInvalidValue;  // stages read the binary32 copy of the state
  if (a.ke_partials) return launch_fused_t<f32x2, float, float, 8, false, true>(a, c, s);
  return launch_fused_t<f32x2, float, float, 8, false, false>(a, c, s);
}

}  // namespace sbli
