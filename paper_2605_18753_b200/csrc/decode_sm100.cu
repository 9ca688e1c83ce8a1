// Stage 2, decode, on tensor cores: shapes served, cluster sizes and launches (kernel: decode_sm100_kernel.cuh).
#include "decode_sm100_kernel.cuh"

namespace dash {

// Splits needed so that no thread block owns more sub-blocks than its list holds (0: shape not served here).
int decode_sm100_min_splits(const Dims& dm) {
  if (!dm.decode || dm.dtype != DASH_BF16 || (dm.d != 64 && dm.d != 128)) return 0;
  if (dm.B != 16 && dm.B != 32 && dm.B != 64 && dm.B != 128) return 0;
  if (dm.qs[2] % 8 != 0 || tensor_map_encoder() == nullptr) return 0;
  if (broadcasts(dm.ks, dm.batch, dm.seq_kv, dm.h_kv) || broadcasts(dm.vs, dm.batch, dm.seq_kv, dm.h_kv)) return 0;
  if (dm.B < SUB) {
    const int cps = SUB / dm.B, range = max_range(dm.g_q) / cps;
    const int max_items = (dm.T_s + cps - 1) / cps + 1;
    return (max_items + range - 1) / range;
  }
  const int max_items = (dm.T_s + 1) * (dm.B / SUB), range = max_range(dm.g_q);
  return (max_items + range - 1) / range;
}

cudaError_t launch_decode_sm100(const Dims& dm, int n_split, const void* Q, const void* K, const void* V,
                                const int* kv_len, const int* count, const int* blk_idx, const float* blk_bias,
                                float* partials, void* O, StatusBlock* sb, cudaStream_t st) {
  DecodeArgs a = {};
  a.O = (__nv_bfloat16*)O;
  a.dm = dm; a.n_split = n_split; a.kv_len = kv_len; a.count = count; a.blk_idx = blk_idx; a.blk_bias = blk_bias;
  a.Q = (const __nv_bfloat16*)Q; a.partials = partials; a.sb = sb;
  // Every block at once: more and shorter splits are the shorter chain, and every group keeps the grid's.  In waves, what a block
  // costs beside its share counts.  (The separate merge kernel, O null, reads every split's slot.)
  a.resident = 2 * current_sm_count();
  const bool waves = (long long)n_split * dm.batch * dm.h_kv > a.resident;
  a.least = O && waves ? 8 : 0;
  if (a.least == 0) a.resident = 1 << 30;
  return launch_any<0>(a, K, V, st);
}

// Blocks per cluster of the fused step (0: not taken): the most of 8, 4, 2 with which the grid is no larger than two blocks per
// SM.  (A measured line: a cluster sits inside one GPC, so the last few of that many clusters may have to wait for others.)  In
// a second wave nothing hides a cluster's serial parts: 104 groups of 4671 tokens take 19 us
// as two kernels and would take 31 in three waves of clusters of eight.  A block's share of the longest possible list is
// bounded as well: lists differ in length, and one long list in two shares is what the step waits for (39 sequences of
// 33597 tokens, 2 KV heads, chunks of 128: 92 us as two kernels, 138 in clusters of two).
static int fused_cluster(const Dims& dm) {
  const int need = decode_sm100_min_splits(dm);
  if (need == 0 || dm.T_s < 1 || dm.T_s > FUSED_MAX_CHUNKS) return 0;
  const int most = dm.T_s * (dm.B > SUB ? dm.B / SUB : 1) / (dm.B < SUB ? SUB / dm.B : 1);     // sub-blocks of the longest list
  for (int cs = 8; cs >= 2 && cs >= need; cs /= 2)
    if ((long long)dm.batch * dm.h_kv * cs <= 2 * current_sm_count()) return most <= 128 * cs ? cs : 0;
  return 0;
}
bool decode_fused_supported(const Dims& dm) { return fused_cluster(dm) > 0; }

cudaError_t launch_decode_fused(const Dims& dm, const void* Q, const void* K, const void* V, const float* Kbar, const int* kv_len,
                                void* O, StatusBlock* sb, cudaStream_t st) {
  DecodeArgs a = {};
  a.O = (__nv_bfloat16*)O;
  a.dm = dm; a.Kbar = Kbar; a.kv_len = kv_len; a.Q = (const __nv_bfloat16*)Q; a.sb = sb;
  switch (fused_cluster(dm)) {
    case 8: return launch_decode_cluster8(a, K, V, st);
    case 4: return launch_decode_cluster4(a, K, V, st);
    case 2: return launch_decode_cluster2(a, K, V, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace dash
