// Stage 1 on tensor cores for sm_100a: bands of tiles by candidate count, and the small kernels around the routing kernel
// (select_sm100_band.cuh).
#include "select_sm100.cuh"
#include "tensor_map.cuh"

namespace dash {

namespace {

__global__ void kbar_split_kernel(const float* __restrict__ kbar, __nv_bfloat16* __restrict__ planes, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  chain_wait();
  chain_release();
  if (i >= n) return;
  const float x = kbar[i];
  const __nv_bfloat16 hi = __float2bfloat16_rn(x);
  const float r1 = x - __bfloat162float(hi);
  const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
  const float r2 = r1 - __bfloat162float(mid);
  planes[i] = hi;
  planes[n + i] = mid;
  planes[2 * n + i] = __float2bfloat16_rn(r2);
}

}  // namespace

// Tokens [0, select_sm100_token_limit) can be routed by the tensor-core kernel (0: not applicable).  A block
// holds 512 candidates per row in tensor memory; clusters of 2 or 4 blocks extend that to 1024 / 2048.
int select_sm100_token_limit(const Dims& dm) {
  if (dm.decode || !dm.causal || dm.dtype != DASH_BF16 || (dm.d != 64 && dm.d != 128) || dm.T_s < 1) return 0;
  if (tensor_map_encoder() == nullptr || broadcasts(dm.qs, dm.batch, dm.seq_q, dm.h_q)) return 0;
  // own chunk index <= 2048, in whole tiles
  const int tq = 128 / dm.g_q;
  const long long lim = (long long)(SELECT_MAX_CS * SELECT_CLUSTER_COLS + 1) * dm.B / tq * tq;
  return (int)(lim < dm.seq_q ? lim : dm.seq_q);
}

size_t select_sm100_scratch_bytes(const Dims& dm) {
  return (size_t)3 * dm.batch * dm.h_kv * (size_t)(dm.T_s > 0 ? dm.T_s : 1) * dm.d * sizeof(__nv_bfloat16);
}

// Local window: the chunks [c_own - L, c_own) of every row are attended with bias 0 without being scored.  The
// routing kernel above leaves them out; this one (launched behind it only when L > 0) sets their mask bits,
// appends them to the row's list behind the routed chunks and adds them to the count.  One thread per row.
__global__ void __launch_bounds__(256)
window_rows_kernel(Dims dm, int token_limit, uint32_t* __restrict__ mask, int* __restrict__ count,
                   int* __restrict__ blk_idx, float* __restrict__ blk_bias) {
  chain_wait();
  chain_release();
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long total = (long long)dm.batch * dm.h_kv * token_limit;
  if (idx >= total) return;
  const int i = (int)(idx % token_limit);
  const long long grp = idx / token_limit;
  const int n_vis = min(i / dm.B, dm.T_s);
  const int n_cand = max(n_vis - dm.local_blocks, 0);
  if (n_vis == n_cand) return;
  const long long row_id = grp * dm.seq_q + i;
  uint32_t* mrow = mask + row_id * dm.W;
  const int routed = count[row_id];
  const long long loff = grp * dm.list_rows + list_row_offset(dm, i) + routed;
  for (int c = n_cand; c < n_vis; ++c) {
    mrow[c >> 5] |= 1u << (c & 31);
    blk_bias[loff + (c - n_cand)] = 0.f;
    if (blk_idx) blk_idx[loff + (c - n_cand)] = c;
  }
  count[row_id] = routed + (n_vis - n_cand);
}

cudaError_t launch_select_sm100(const Dims& dm, int token_limit, const void* Q, const float* Kbar, void* planes,
                                uint32_t* mask, int* count, int* blk_idx, float* blk_bias, float* tau,
                                StatusBlock* sb, cudaStream_t st, bool planes_ready) {
  const long long plane_rows = (long long)dm.batch * dm.h_kv * dm.T_s;
  const long long n = plane_rows * dm.d;
  cudaError_t e = cudaSuccess;
  if (!planes_ready) {       // the summaries came from the caller: split them here
    e = launch_chained(kbar_split_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, Kbar,
                       (__nv_bfloat16*)planes, n);
    count_launch();
    if (e != cudaSuccess) return e;
  }

  SelectTcArgs a;
  a.dm = dm;
  a.TQ = 128 / dm.g_q;
  a.plane_rows = plane_rows;
  a.mask = mask; a.count = count; a.blk_idx = blk_idx; a.blk_bias = blk_bias; a.tau = tau; a.sb = sb;

  CUtensorMap tq, tkb;
  {
    cuuint64_t dims[4] = {(cuuint64_t)dm.d, (cuuint64_t)dm.h_q, (cuuint64_t)dm.seq_q, (cuuint64_t)dm.batch};
    auto sb2 = [](long long el) { return (cuuint64_t)((el > 0 ? el : 8) * 2); };
    cuuint64_t strides[3] = {sb2(dm.qs[2]), sb2(dm.qs[1]), sb2(dm.qs[0])};
    cuuint32_t box[4] = {64u, (cuuint32_t)dm.g_q, (cuuint32_t)a.TQ, 1u};
    if (!encode_bf16_sw128_4d(&tq, Q, dims, strides, box)) return cudaErrorInvalidValue;
  }
  {
    const cuuint64_t hd = (cuuint64_t)dm.d;
    cuuint64_t dims[4] = {hd, (cuuint64_t)(3 * plane_rows), 1, 1};
    cuuint64_t strides[3] = {hd * 2, (cuuint64_t)(3 * plane_rows) * hd * 2, (cuuint64_t)(3 * plane_rows) * hd * 2};
    cuuint32_t box[4] = {64u, (cuuint32_t)SELECT_SC, 1u, 1u};
    if (!encode_bf16_sw128_4d(&tkb, planes, dims, strides, box)) return cudaErrorInvalidValue;
  }
  // Bands of tiles by candidate count: <= 512 one block per tile, <= 1024 clusters of 2, <= 2048 clusters of 4.
  // Tiles are TQ tokens; a tile's candidate count is the own chunk index of its last token.
  const auto shorter = dm.d == 64 ? select_band_d64_short : select_band_d128_short;
  const auto longer = dm.d == 64 ? select_band_d64_long : select_band_d128_long;
  const int groups = dm.batch * dm.h_kv;
  const int total_tiles = (token_limit + a.TQ - 1) / a.TQ;
  auto tiles_up_to = [&](long long max_cand) -> int {      // tiles whose own chunk indexes are all <= max_cand
    const long long tokens = (max_cand + 1) * dm.B;
    const long long t = tokens / a.TQ;
    return (int)(t < total_tiles ? t : total_tiles);
  };
  const int t1 = tiles_up_to(SELECT_CLUSTER_COLS), t2 = tiles_up_to(2 * SELECT_CLUSTER_COLS), t3 = total_tiles;
  // widest bands first: they are the long-running ones
  if (t3 > t2) {
    a.tile_base = t2; a.n_tiles = t3 - t2; a.tmem_cols = 512;
    if ((e = longer(dm, 4, tq, tkb, a, (long long)a.n_tiles * groups, st)) != cudaSuccess) return e;
  }
  if (t2 > t1) {
    a.tile_base = t1; a.n_tiles = t2 - t1; a.tmem_cols = 512;
    if ((e = longer(dm, 2, tq, tkb, a, (long long)a.n_tiles * groups, st)) != cudaSuccess) return e;
  }
  // one block per tile: rows of 257 .. 512 candidates take the whole tensor memory of an SM (one block per SM, three
  // solver threads per row); shorter ones leave room for two blocks per SM with the row in one thread
  const int t0 = tiles_up_to(256);
  if (t1 > t0) {
    a.tile_base = t0; a.n_tiles = t1 - t0; a.tmem_cols = 512;
    if ((e = longer(dm, 1, tq, tkb, a, (long long)a.n_tiles * groups, st)) != cudaSuccess) return e;
  }
  {
    a.tile_base = 0; a.n_tiles = t0;
    const int max_cand = min(dm.T_s, (int)(((long long)t0 * a.TQ - 1) / dm.B));
    uint32_t cols = 32;
    while ((int)cols < ((max_cand + SELECT_SC - 1) / SELECT_SC) * SELECT_SC) cols <<= 1;
    a.tmem_cols = cols;
    e = shorter(dm, 1, tq, tkb, a, (long long)a.n_tiles * groups, st);
  }
  if (e == cudaSuccess && dm.local_blocks > 0) {
    const long long rows = (long long)groups * token_limit;
    e = launch_chained(window_rows_kernel, dim3((unsigned)((rows + 255) / 256)), dim3(256), 0, st, dm, token_limit,
                       mask, count, blk_idx, blk_bias);
    count_launch();
  }
  return e;
}

}  // namespace dash
