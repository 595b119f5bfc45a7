// FP64 instances of the fused kernel with every block update at k = 4 in
// register form, blocks three nodes wide (even d) included.
#include "bbp_decode_inst.cuh"

namespace bbp {

cudaError_t launch_fused_any_f64(const LaunchArgs& a, int warps, int cosets, int lean, cudaStream_t st) {
  switch (warps * 1000 + cosets * 100 + lean) {
    case 16111: return launch_fused_nw<double, 16, 1, 4, false, 11>(a, st);
    case 16211: return launch_fused_nw<double, 16, 2, 4, false, 11>(a, st);
    case 8411: return launch_fused_nw<double, 8, 4, 4, false, 11>(a, st);
    case 8212: return launch_fused_nw<double, 8, 2, 4, false, 12>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_fused_mixed_any_f64(const LaunchArgs& a, const MixedLaunch& m, int warps, int cosets, int lean,
                                       cudaStream_t st) {
  switch (warps * 1000 + cosets * 100 + lean) {
    case 16111: return launch_fused_mixed_nw<double, 16, 1, 4, false, 11>(a, m, st);
    case 16211: return launch_fused_mixed_nw<double, 16, 2, 4, false, 11>(a, m, st);
    case 8411: return launch_fused_mixed_nw<double, 8, 4, 4, false, 11>(a, m, st);
    case 8212: return launch_fused_mixed_nw<double, 8, 2, 4, false, 12>(a, m, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace bbp
