// Instantiations of the fused scoring kernel: head dimension 64, bf16 keys.
#include "fused.cuh"

namespace spf {
int32_t fused_launch_d64(const FusedArgs& args, const FusedLaunch& l, cudaStream_t stream) { return fused_launch<64, false>(args, l, stream); }
}  // namespace spf
