// Stage 1 for decode (Eq. 2, Eq. 4, Algorithm 2, Proposition 1): one query row per sequence.
//
// Decode routing is HBM-bound on the summary cache (every candidate's kbar row is read once per step and per KV head).
// Caches of up to 512 chunks take one kernel, one block per (batch, KV head):
//   decode_select_kernel  streams kbar with fully coalesced row reads (one warp per row, several rows in flight), keeps the
//                         scaled chunk logits x = gamma(alpha-1) <q, kbar_c>/sqrt(d) of the g_q heads in shared memory and
//                         routes the group (decode_route.cuh).  Two to four blocks per SM: one group's routing, which moves
//                         nothing, passes under other groups' streams.
// Longer caches are split in two:
//   decode_scores_kernel  many thread blocks per (batch, KV head) write the logits to a small fp32 scratch (b * h_q * T_s
//                         floats, stays in L2);
//   decode_route_kernel   one thread block of 16 warps per (batch, KV head) loads its g_q logit rows into shared memory and
//                         routes the group.
// With a local window of L chunks the last L chunks before the own one are not scored; routing sets their bits and appends
// them to the list with bias 0.
#include "decode_route.cuh"

namespace dash {

namespace {

constexpr int SC_WARPS = 8;
constexpr int SC_ROWS_PER_BLOCK = 256;   // summary rows one thread block scores
constexpr int RT_THREADS = 512;      // 128 registers per thread: a Newton warp keeps 64 logits per lane in registers
constexpr int RT_LOADS = 4;           // logits per head a thread requests per sweep (2048 candidates: one sweep)
constexpr int SL_MAX_CHUNKS = 512;    // a Newton warp keeps 16 logits per lane: 64 registers, four blocks per SM

struct RouteOut {
  uint32_t* mask;
  int* count;
  int* blk_idx;
  float* blk_bias;
  float* tau;
};

// The row's lists, mask words and count in global memory, from logits in shared memory.
template <int G, int NW, int MAXR>
__device__ __forceinline__ void route_to_global(const Dims& dm, float* X, int stride, int n_cand, int n_vis, int c_own, float* taus,
                                                float* wsum, int* wcnt, const RouteOut& o, int b, int r, int warp, int lane) {
  const long long grp = (long long)b * dm.h_kv + r, loff = grp * dm.list_rows;
  uint32_t* mrow = o.mask + grp * dm.W;
  route_group<G, NW, MAXR>(dm, X, stride, n_cand, n_vis, dm.W, taus, wsum, wcnt, warp, lane,
                           [&](int j, uint32_t word) { mrow[j] = word | (((c_own >> 5) == j) ? (1u << (c_own & 31)) : 0u); },
                           [&](int n) {
                             if (warp == 0 && lane == 0) o.count[grp] = n;
                             if (o.tau && warp == 0 && lane < G) o.tau[(long long)b * dm.h_q + r * G + lane] = taus[lane];
                           },
                           [&](int pos, int c, float bias) {
                             o.blk_bias[loff + pos] = bias;
                             if (o.blk_idx) o.blk_idx[loff + pos] = c;
                           });
}

template <typename T, int D, int G, int NW>
__global__ void __launch_bounds__(NW * 32, (G * D <= 1024 ? 32 : 16) / NW)
decode_select_kernel(Dims dm, const T* __restrict__ Q, const float* __restrict__ Kbar, const int* __restrict__ kv_len, RouteOut out) {
  extern __shared__ __align__(16) float sm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r = blockIdx.x, b = blockIdx.y;
  warm_length(kv_len, b);
  chain_wait();
  chain_release();
  const int L = sequence_length(dm, kv_len, b);
  const int c_own = (L - 1) >> dm.log_b;
  const int n_vis = min(c_own, dm.T_s);                 // chunks before the own one: candidates, then the window
  const int n_cand = max(n_vis - dm.local_blocks, 0);   // scored by entmax
  const int stride = route_stride(n_vis);
  float* X = sm;                                 // [G][stride] all logits of the group
  float* taus = X + (size_t)G * stride;          // [G] (32 floats reserved)
  float* wsum = taus + 32;
  int* wcnt = reinterpret_cast<int*>(wsum + dm.W);
  if (n_cand > 0) {
    float q[G][D / 32];
    load_query<T, D, G>(dm, Q, b, r, lane, q);
    const float* kb = Kbar + ((long long)b * dm.h_kv + r) * dm.T_s * D + lane * (D / 32);
    score_rows<D, G>(q, kb, 0, n_cand, warp, NW, lane, [&](int g, int c, float x) { X[(size_t)g * stride + c] = x; });
  }
  __syncthreads();
  route_to_global<G, NW, 16>(dm, X, stride, n_cand, n_vis, c_own, taus, wsum, wcnt, out, b, r, warp, lane);
}

template <typename T, int D, int G>
__global__ void __launch_bounds__(SC_WARPS * 32)
decode_scores_kernel(Dims dm, const T* __restrict__ Q, const float* __restrict__ Kbar, const int* __restrict__ kv_len,
                     float* __restrict__ xs) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r = blockIdx.y, b = blockIdx.z;
  warm_length(kv_len, b);
  chain_wait();
  chain_release();
  const int L = sequence_length(dm, kv_len, b);
  const int n_cand = max(min((L - 1) >> dm.log_b, dm.T_s) - dm.local_blocks, 0);   // window chunks are not scored
  const int c_begin = blockIdx.x * SC_ROWS_PER_BLOCK;
  const int c_end = min(n_cand, c_begin + SC_ROWS_PER_BLOCK);
  if (c_begin >= c_end) return;
  float q[G][D / 32];
  load_query<T, D, G>(dm, Q, b, r, lane, q);
  const float* kb = Kbar + ((long long)b * dm.h_kv + r) * dm.T_s * D + lane * (D / 32);
  float* xo = xs + ((long long)b * dm.h_kv + r) * G * dm.T_s;
  score_rows<D, G>(q, kb, c_begin, c_end, warp, SC_WARPS, lane, [&](int g, int c, float x) { xo[(long long)g * dm.T_s + c] = x; });
}

template <int G>
__global__ void __launch_bounds__(RT_THREADS)
decode_route_kernel(Dims dm, const float* __restrict__ xs, const int* __restrict__ kv_len, RouteOut out) {
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r = blockIdx.x, b = blockIdx.y;
  warm_length(kv_len, b);
  chain_wait();
  chain_release();
  const int L = sequence_length(dm, kv_len, b);
  const int c_own = (L - 1) >> dm.log_b;
  const int n_vis = min(c_own, dm.T_s);
  const int n_cand = max(n_vis - dm.local_blocks, 0);
  const int stride = route_stride(n_vis);
  float* X = sm;
  float* taus = X + (size_t)G * stride;
  float* wsum = taus + 32;
  int* wcnt = reinterpret_cast<int*>(wsum + dm.W);
  const float* xg = xs + ((long long)b * dm.h_kv + r) * G * dm.T_s;
  // all of a thread's loads of one sweep are issued before the first is used (one L2 round trip per sweep)
  for (int c0 = 0; c0 < n_cand; c0 += RT_LOADS * RT_THREADS) {
    float v[G][RT_LOADS];
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int u = 0; u < RT_LOADS; ++u) {
        const int c = c0 + u * RT_THREADS + tid;
        if (c < n_cand) v[g][u] = __ldcg(xg + (long long)g * dm.T_s + c);
      }
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int u = 0; u < RT_LOADS; ++u) {
        const int c = c0 + u * RT_THREADS + tid;
        if (c < n_cand) X[(size_t)g * stride + c] = v[g][u];
      }
  }
  __syncthreads();
  route_to_global<G, RT_THREADS / 32, 64>(dm, X, stride, n_cand, n_vis, c_own, taus, wsum, wcnt, out, b, r, warp, lane);
}

}  // namespace

size_t select_decode_scratch_bytes(const Dims& dm) {
  return dm.decode ? (size_t)dm.batch * dm.h_q * (size_t)(dm.T_s > 0 ? dm.T_s : 1) * sizeof(float) : 0;
}

static size_t route_smem(const Dims& dm) {
  // logits, taus, per-word sums and counts
  return ((size_t)dm.g_q * route_stride(dm.T_s) + 32 + dm.W + dm.W + 1 + 8) * sizeof(float);
}

bool select_decode_supported(const Dims& dm) { return dm.decode && route_smem(dm) <= 200 * 1024; }

template <typename T, int D, int G>
static cudaError_t launch_group_size(const Dims& dm, const void* Q, const float* Kbar, const int* kv_len, const RouteOut& out,
                                     float* scratch, cudaStream_t st) {
  const size_t smem = route_smem(dm);
  // one block per group up to 512 chunks: a launch and the logits' way through L2 saved
  // (sixteen warps instead of eight where rows are long: a row is one block's chain of loads)
  if (dm.T_s <= SL_MAX_CHUNKS) {
    const dim3 grid(dm.h_kv, dm.batch);
    cudaError_t e = dm.T_s > SL_MAX_CHUNKS / 4
                        ? launch_chained(decode_select_kernel<T, D, G, 16>, grid, dim3(16 * 32), smem, st, dm, (const T*)Q, Kbar, kv_len, out)
                        : launch_chained(decode_select_kernel<T, D, G, 8>, grid, dim3(8 * 32), smem, st, dm, (const T*)Q, Kbar, kv_len, out);
    count_launch();
    return e;
  }
  const int blocks_x = (dm.T_s + SC_ROWS_PER_BLOCK - 1) / SC_ROWS_PER_BLOCK;
  cudaError_t e = launch_chained(decode_scores_kernel<T, D, G>, dim3(blocks_x, dm.h_kv, dm.batch), dim3(SC_WARPS * 32), 0, st, dm,
                                 (const T*)Q, Kbar, kv_len, scratch);
  count_launch();
  if (e != cudaSuccess) return e;
  static std::atomic<unsigned long long> configured{0};
  if ((e = allow_dynamic_smem(decode_route_kernel<G>, 200 * 1024, configured)) != cudaSuccess) return e;
  e = launch_chained(decode_route_kernel<G>, dim3(dm.h_kv, dm.batch), dim3(RT_THREADS), smem, st, dm, (const float*)scratch, kv_len, out);
  count_launch();
  return e;
}

cudaError_t launch_select_decode(const Dims& dm, const void* Q, const float* Kbar, const int* kv_len, uint32_t* mask,
                                 int* count, int* blk_idx, float* blk_bias, float* tau, float* scratch,
                                 cudaStream_t st) {
  const RouteOut out = {mask, count, blk_idx, blk_bias, tau};
#define DASH_SC_G(T, D)                                                                           \
  switch (dm.g_q) {                                                                               \
    case 1: return launch_group_size<T, D, 1>(dm, Q, Kbar, kv_len, out, scratch, st);             \
    case 2: return launch_group_size<T, D, 2>(dm, Q, Kbar, kv_len, out, scratch, st);             \
    case 4: return launch_group_size<T, D, 4>(dm, Q, Kbar, kv_len, out, scratch, st);             \
    case 8: return launch_group_size<T, D, 8>(dm, Q, Kbar, kv_len, out, scratch, st);             \
    case 16: return launch_group_size<T, D, 16>(dm, Q, Kbar, kv_len, out, scratch, st);           \
    default: return cudaErrorInvalidValue;                                                        \
  }
  if (dm.dtype == DASH_BF16) {
    if (dm.d == 128) { DASH_SC_G(__nv_bfloat16, 128) } else { DASH_SC_G(__nv_bfloat16, 64) }
  } else {
    if (dm.d == 128) { DASH_SC_G(float, 128) } else { DASH_SC_G(float, 64) }
  }
#undef DASH_SC_G
}

}  // namespace dash
