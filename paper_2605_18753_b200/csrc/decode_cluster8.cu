// The fused decode step in clusters of 8 blocks (see decode_sm100_kernel.cuh).
#include "decode_sm100_kernel.cuh"

namespace dash {
cudaError_t launch_decode_cluster8(DecodeArgs& a, const void* K, const void* V, cudaStream_t st) { return launch_any<8>(a, K, V, st); }
}  // namespace dash
