// FP32 instances of the fused kernel with every block update at k = 4 in
// register form, blocks three nodes wide (even d) included.
#include "bbp_decode_inst.cuh"

namespace bbp {

cudaError_t launch_fused_any_f32(const LaunchArgs& a, int warps, int cosets, int lean, cudaStream_t st) {
  switch (warps * 1000 + cosets * 100 + lean) {
    case 16111: return launch_fused_nw<float, 16, 1, 4, false, 11>(a, st);
    case 16211: return launch_fused_nw<float, 16, 2, 4, false, 11>(a, st);
    case 16411: return launch_fused_nw<float, 16, 4, 4, false, 11>(a, st);
    case 8412: return launch_fused_nw<float, 8, 4, 4, false, 12>(a, st);
    case 8413: return launch_fused_nw<float, 8, 4, 4, false, 13>(a, st);
    case 8414: return launch_fused_nw<float, 8, 4, 4, false, 14>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_fused_mixed_any_f32(const LaunchArgs& a, const MixedLaunch& m, int warps, int cosets, int lean,
                                       cudaStream_t st) {
  switch (warps * 1000 + cosets * 100 + lean) {
    case 16111: return launch_fused_mixed_nw<float, 16, 1, 4, false, 11>(a, m, st);
    case 16211: return launch_fused_mixed_nw<float, 16, 2, 4, false, 11>(a, m, st);
    case 16411: return launch_fused_mixed_nw<float, 16, 4, 4, false, 11>(a, m, st);
    case 8412: return launch_fused_mixed_nw<float, 8, 4, 4, false, 12>(a, m, st);
    case 8413: return launch_fused_mixed_nw<float, 8, 4, 4, false, 13>(a, m, st);
    case 8414: return launch_fused_mixed_nw<float, 8, 4, 4, false, 14>(a, m, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace bbp
