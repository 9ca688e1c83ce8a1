// The fused decode step in clusters of 4 blocks (see decode_sm100_kernel.cuh).
#include "decode_sm100_kernel.cuh"

namespace dash {
cudaError_t launch_decode_cluster4(DecodeArgs& a, const void* K, const void* V, cudaStream_t st) { return launch_any<4>(a, K, V, st); }
}  // namespace dash
