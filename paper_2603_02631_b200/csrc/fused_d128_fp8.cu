// Instantiations of the fused scoring kernel: head dimension 128, E4M3 keys.
#include "fused.cuh"

namespace spf {
int32_t fused_launch_d128_fp8(const FusedArgs& args, const FusedLaunch& l, cudaStream_t stream) { return fused_launch<128, true>(args, l, stream); }
}  // namespace spf
