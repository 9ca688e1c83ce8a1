// Stage 2, prefill, CUDA-core path (Eq. 7 in the form of Proposition 1; Algorithm 3): fp32 tensors and the non-causal
// mode.
//
// Tile: AG_ROWS consecutive (token, head-of-group) rows of one (batch, KV head), token-major; a tile never straddles a
// chunk.  A block's eight warps share the tile's walk over the union of its rows' chunks, 32 keys at a time, slice k going
// to warp k mod 8; every warp keeps the online softmax (m, l, O) of all rows over its slices and the block merges the
// eight states in shared memory at the end.  Inside a slice lanes own keys for the logits (a lane's key row is read once
// for all rows; queries come from shared memory as broadcasts) and head_dim slices for the output (a value row is read once
// for all rows, the probabilities are broadcasts).  A row that did not route a chunk gets bias -inf there.
// Bound by FFMA issue for large problems and by the length of the longest row's walk for small ones; eight rows per key
// load and eight warps per walk serve both ends (one warp per row, as it was: 1024 tokens, one head, d 64: 82 us, now 9).
#include "common.cuh"
#include "tile_walk.cuh"

namespace dash {

constexpr int AG_WARPS = 8;
constexpr int AG_ROWS = 8;

template <typename T, int D>
__global__ void __launch_bounds__(AG_WARPS * 32, 2)
attend_prefill_generic_kernel(Dims dm, int n_tiles, const T* __restrict__ Q, const T* __restrict__ K, const T* __restrict__ V,
                              const uint32_t* __restrict__ mask, const float* __restrict__ blk_bias,
                              T* __restrict__ O) {
  constexpr int VPL = D / 32, R = AG_ROWS;
  __shared__ __align__(16) float qs[R][D];
  __shared__ __align__(16) float ps[AG_WARPS][32][R];
  __shared__ float ml[AG_WARPS][R][2];
  __shared__ float part[R][D];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int groups = dm.batch * dm.h_kv;
  const int tile = n_tiles - 1 - (int)(blockIdx.x / groups);      // long rows first
  const int grp = (int)(blockIdx.x % groups), b = grp / dm.h_kv, r = grp % dm.h_kv;
  const int row0 = tile * R;                                      // row = token * g_q + head of the group
  const int n_rows = min(R, dm.seq_q * dm.g_q - row0);
  const int i0 = row0 / dm.g_q, n_tok = (row0 + n_rows - 1) / dm.g_q - i0 + 1;
  const int c_own = dm.causal ? i0 >> dm.log_b : dm.T_s;   // non-causal: the incomplete tail chunk, seen whole by every row
  chain_wait();
  chain_release();

  for (int idx = threadIdx.x; idx < R * D; idx += AG_WARPS * 32) {
    const int rr = idx / D, k = idx % D, row = row0 + rr, i = row / dm.g_q, h = r * dm.g_q + row % dm.g_q;
    qs[rr][k] = rr < n_rows ? to_f32<T>(Q[(long long)b * dm.qs[0] + (long long)i * dm.qs[1] + (long long)h * dm.qs[2] + k]) * dm.sm_scale : 0.f;
  }
  __syncthreads();

  const T* kbase = K + (long long)b * dm.ks[0] + (long long)r * dm.ks[2];
  const T* vbase = V + (long long)b * dm.vs[0] + (long long)r * dm.vs[2] + lane * VPL;
  // lane t < n_tok looks after token i0 + t: its mask word, routed chunks so far, list
  const int my_tok = min(lane, n_tok - 1);
  const uint32_t* mrow = mask + ((long long)grp * dm.seq_q + i0 + my_tok) * dm.W;
  const float* list = blk_bias + (long long)grp * dm.list_rows + list_row_offset(dm, i0 + my_tok);

  float m[R], l[R], acc[R][VPL];
#pragma unroll
  for (int rr = 0; rr < R; ++rr) {
    m[rr] = -INFINITY;
    l[rr] = 0.f;
#pragma unroll
    for (int v = 0; v < VPL; ++v) acc[rr][v] = 0.f;
  }
  int slice = 0, seen = 0;
  for (int w = 0; w <= (min(c_own, dm.T_a - 1) >> 5); ++w) {
    const uint32_t routed = lane < n_tok ? routed_bits(mrow[w], w, c_own) : 0u;
    uint32_t u = __reduce_or_sync(0xffffffffu, routed);
    if ((c_own >> 5) == w && c_own < dm.T_a) u |= 1u << (c_own & 31);     // attended by every row
    while (u != 0u) {
      const int bit = __ffs(u) - 1, c = w * 32 + bit;
      u &= u - 1;
      const bool own = c == c_own;
      const int t_beg = c << dm.log_b, t_stop = own && dm.causal ? i0 + n_tok : min(t_beg + dm.B, dm.seq_kv);
      const int n_sl = (t_stop - t_beg + 31) >> 5;
      const int first = (warp - slice) & (AG_WARPS - 1);                  // this warp's first slice of the chunk
      slice += n_sl;
      if (first >= n_sl) continue;
      float bias = own ? 0.f : -INFINITY;
      if (!own && ((routed >> bit) & 1u)) bias = list[seen + __popc(routed & ((1u << bit) - 1u))];
      for (int sl = first; sl < n_sl; sl += AG_WARPS) {
        const int t0 = t_beg + sl * 32, t = t0 + lane;
        float s[R];
#pragma unroll
        for (int rr = 0; rr < R; ++rr) s[rr] = 0.f;
        const T* kp = kbase + (long long)min(t, dm.seq_kv - 1) * dm.ks[1];
#pragma unroll 4
        for (int k = 0; k < D; k += 4) {
          const float4 kv = load4(kp + k);
#pragma unroll
          for (int rr = 0; rr < R; ++rr) {
            const float4 qv = *reinterpret_cast<const float4*>(&qs[rr][k]);
            s[rr] = fmaf(qv.x, kv.x, s[rr]); s[rr] = fmaf(qv.y, kv.y, s[rr]);
            s[rr] = fmaf(qv.z, kv.z, s[rr]); s[rr] = fmaf(qv.w, kv.w, s[rr]);
          }
        }
#pragma unroll
        for (int rr = 0; rr < R; ++rr) {
          const int i = (row0 + rr) / dm.g_q;
          const float bv = __shfl_sync(0xffffffffu, bias, min(i - i0, n_tok - 1));
          const bool vis = t < t_stop && !(own && dm.causal && t > i);
          const float x = vis ? s[rr] + bv : -INFINITY;
          const float mt = fmaxf(m[rr], warp_max(x));
          // (a row that has seen nothing yet keeps m = -inf: its corrections and probabilities are 0, not NaN)
          const float corr = mt > -INFINITY ? __expf(m[rr] - mt) : 1.f;
          const float p = x > -INFINITY ? __expf(x - mt) : 0.f;
          l[rr] = l[rr] * corr + p;                 // per-lane partial sum; reduced across lanes at the end
#pragma unroll
          for (int v = 0; v < VPL; ++v) acc[rr][v] *= corr;
          m[rr] = mt;
          ps[warp][lane][rr] = p;
        }
        __syncwarp();
        const int nt = min(32, t_stop - t0);
#pragma unroll 4
        for (int q = 0; q < nt; ++q) {
          float vv[VPL];
          const T* vp = vbase + (long long)(t0 + q) * dm.vs[1];
          if constexpr (VPL == 4) {
            const float4 f = load4(vp);
            vv[0] = f.x; vv[1] = f.y; vv[2] = f.z; vv[3] = f.w;
          } else {
            vv[0] = to_f32<T>(vp[0]); vv[1] = to_f32<T>(vp[1]);
          }
          const float4 pa = *reinterpret_cast<const float4*>(&ps[warp][q][0]), pb = *reinterpret_cast<const float4*>(&ps[warp][q][4]);
          const float pr[R] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
#pragma unroll
          for (int rr = 0; rr < R; ++rr)
#pragma unroll
            for (int v = 0; v < VPL; ++v) acc[rr][v] = fmaf(pr[rr], vv[v], acc[rr][v]);
        }
        __syncwarp();
      }
    }
    seen += __popc(routed);
  }

  // merge: every warp brings its state onto the block's maximum, the outputs are added in warp order
#pragma unroll
  for (int rr = 0; rr < R; ++rr) {
    const float ls = warp_sum(l[rr]);
    if (lane == 0) { ml[warp][rr][0] = m[rr]; ml[warp][rr][1] = ls; }
  }
  __syncthreads();
  float wgt[R];
#pragma unroll
  for (int rr = 0; rr < R; ++rr) {
    float M = -INFINITY;
#pragma unroll
    for (int q = 0; q < AG_WARPS; ++q) M = fmaxf(M, ml[q][rr][0]);
    float tot = 0.f;
#pragma unroll
    for (int q = 0; q < AG_WARPS; ++q) tot += ml[q][rr][0] > -INFINITY ? ml[q][rr][1] * __expf(ml[q][rr][0] - M) : 0.f;
    wgt[rr] = m[rr] > -INFINITY && tot > 0.f ? __expf(m[rr] - M) / tot : 0.f;
  }
  for (int q = 0; q < AG_WARPS; ++q) {
    if (warp == q) {
#pragma unroll
      for (int rr = 0; rr < R; ++rr)
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
          const float x = acc[rr][v] * wgt[rr];
          if (q == 0) part[rr][lane * VPL + v] = x; else part[rr][lane * VPL + v] += x;
        }
    }
    __syncthreads();
  }
  const int row = row0 + warp;                     // (eight warps, eight rows)
  if (warp < n_rows) {
    T* op = O + (long long)b * dm.os[0] + (long long)(row / dm.g_q) * dm.os[1] + (long long)(r * dm.g_q + row % dm.g_q) * dm.os[2] + lane * VPL;
#pragma unroll
    for (int v = 0; v < VPL; ++v) op[v] = from_f32<T>(part[warp][lane * VPL + v]);
  }
}
static_assert(AG_ROWS == AG_WARPS, "the epilogue writes one row per warp");

cudaError_t launch_attend_prefill_generic(const Dims& dm, const void* Q, const void* K, const void* V,
                                          const uint32_t* mask, const float* blk_bias, void* O, cudaStream_t st) {
  const long long n_tiles = ((long long)dm.seq_q * dm.g_q + AG_ROWS - 1) / AG_ROWS;
  const unsigned grid = (unsigned)(n_tiles * dm.batch * dm.h_kv);
  cudaError_t le = cudaSuccess;
#define DASH_LAUNCH_AG(T, D)                                                                                    \
  le = launch_chained(attend_prefill_generic_kernel<T, D>, dim3(grid), dim3(AG_WARPS * 32), 0, st, dm,          \
                      (int)n_tiles, (const T*)Q, (const T*)K, (const T*)V, mask, blk_bias, (T*)O)
  if (dm.dtype == DASH_BF16) {
    if (dm.d == 128) DASH_LAUNCH_AG(__nv_bfloat16, 128); else DASH_LAUNCH_AG(__nv_bfloat16, 64);
  } else {
    if (dm.d == 128) DASH_LAUNCH_AG(float, 128); else DASH_LAUNCH_AG(float, 64);
  }
#undef DASH_LAUNCH_AG
  count_launch();
  return le;
}

}  // namespace dash
