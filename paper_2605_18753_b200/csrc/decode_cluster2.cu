// The fused decode step in clusters of 2 blocks (see decode_sm100_kernel.cuh).
#include "decode_sm100_kernel.cuh"

namespace dash {
cudaError_t launch_decode_cluster2(DecodeArgs& a, const void* K, const void* V, cudaStream_t st) { return launch_any<2>(a, K, V, st); }
}  // namespace dash
