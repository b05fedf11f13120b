// Instantiations of the fused scoring kernel: head dimension 128, bf16 keys.
#include "fused.cuh"

namespace spf {
int32_t fused_launch_d128(const FusedArgs& args, const FusedLaunch& l, cudaStream_t stream) { return fused_launch<128, false>(args, l, stream); }
}  // namespace spf
