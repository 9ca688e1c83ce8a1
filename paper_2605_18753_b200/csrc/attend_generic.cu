// Stage 2, prefill, CUDA-core path (Eq. 7 in the form of Proposition 1; Algorithm 3): fp32 tensors and the non-causal
// mode.
//
// Tile: R consecutive (token, head-of-group) rows of one (batch, KV head), token-major; a tile never straddles a chunk.
// The block enters the chunks of the tile's union with their biases into shared memory, then its NW warps share them, 32
// keys at a time, slice k going to warp k mod NW; every warp keeps the online softmax (m, l, O) of all rows over its slices
// and the block merges the states in shared memory at the end.  A row that did not route a chunk has bias -inf there.
//
// Inside a slice four lanes share a key row for the logits: lane l reads the 16-byte pieces (l mod 4) + 4 j of the keys
// (l div 4) + 8 k, so that a load touches 8 lines instead of 32 and a query piece read from shared memory serves four keys;
// the four partial sums meet in three shuffles per row, which leave key (l div 4) + 8 * (l mod 4) in lane l.  For the
// output lanes own head_dim slices: a value row is read once for all rows, the probabilities are broadcasts.
// Bound by FFMA issue for large problems (R = 8) and, where there are few tiles, by the chain of the longest tile's walk:
// R = 4 halves it and leaves registers for a whole slice's loads in flight.  1024 tokens, one head, d 64: 82 us with one warp per row,
// now 19; three prompts of 1500, 12 heads: 3 to 5 times faster.
#include "common.cuh"
#include "tile_walk.cuh"

namespace dash {

// Floats of a block's dynamic shared memory: a slice's probabilities per warp in the walk, the warps' outputs at the end.
template <int D, int R, int NW> constexpr int buf_floats() { return NW * R * (D > 32 ? D : 32); }

template <typename T, int D, int R, int NW>
__global__ void __launch_bounds__(NW * 32, 16 / NW)
attend_prefill_generic_kernel(Dims dm, int n_tiles, const T* __restrict__ Q, const T* __restrict__ K, const T* __restrict__ V,
                              const uint32_t* __restrict__ mask, const float* __restrict__ blk_bias,
                              T* __restrict__ O) {
  constexpr int VPL = D / 32;
  constexpr int SEG = 32 * NW;              // chunks entered at a time, one mask word per warp
  __shared__ __align__(16) float qs[R][D];
  extern __shared__ __align__(16) float buf[];
  __shared__ float ml[NW][R][2];
  __shared__ int seg_chunk[SEG], seg_n;
  __shared__ float seg_bias[SEG][R + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int log_g = 31 - __clz(dm.g_q);                           // (group sizes are powers of two)
  const int groups = dm.batch * dm.h_kv;
  const int tile = n_tiles - 1 - (int)(blockIdx.x / groups);      // long rows first
  const int grp = (int)(blockIdx.x % groups), b = grp / dm.h_kv, r = grp % dm.h_kv;
  const int row0 = tile * R;                                      // row = token * g_q + head of the group
  const int n_rows = min(R, dm.seq_q * dm.g_q - row0);
  const int i0 = row0 >> log_g, n_tok = ((row0 + n_rows - 1) >> log_g) - i0 + 1;
  const int c_own = dm.causal ? i0 >> dm.log_b : dm.T_s;   // non-causal: the incomplete tail chunk, seen whole by every row
  chain_wait();
  chain_release();

  for (int idx = threadIdx.x; idx < R * D; idx += NW * 32) {
    const int rr = idx / D, k = idx % D, row = row0 + rr, i = row >> log_g, h = r * dm.g_q + (row & (dm.g_q - 1));
    qs[rr][k] = rr < n_rows ? to_f32<T>(Q[(long long)b * dm.qs[0] + (long long)i * dm.qs[1] + (long long)h * dm.qs[2] + k]) * dm.sm_scale : 0.f;
  }
  const int my_key = (lane >> 2) + 8 * (lane & 3);                // (bit 1 of the lane chose keys + 16, bit 0 keys + 8)
  const T* kbase = K + (long long)b * dm.ks[0] + (long long)r * dm.ks[2] + 4 * (lane & 3);
  const T* vbase = V + (long long)b * dm.vs[0] + (long long)r * dm.vs[2] + lane * VPL;

  float m[R], l[R], acc[R][VPL];
#pragma unroll
  for (int rr = 0; rr < R; ++rr) {
    m[rr] = -INFINITY;
    l[rr] = 0.f;
#pragma unroll
    for (int v = 0; v < VPL; ++v) acc[rr][v] = 0.f;
  }
  float* ps = buf + warp * 32 * R;
  // The union's chunks, SEG at a time: entry = (chunk, bias of every token; -inf: the token does not attend it), the own
  // chunk (bias 0) last of all.  Warp w enters the chunks of mask word w of the segment, lane = chunk.
  const int n_words = (min(c_own, dm.T_a - 1) >> 5) + 1;
  const int spc = dm.B > 32 ? dm.B >> 5 : 1;                      // slices per chunk
  const uint32_t* mrow = mask + ((long long)grp * dm.seq_q + i0) * dm.W;
  for (int w0 = 0; w0 < n_words; w0 += SEG / 32) {
    const int n_w = min(SEG / 32, n_words - w0);
    if (w0 > 0) __syncthreads();          // (the segment before has been walked)
    if (warp < n_w) {
      int before = 0, pos[R];             // entries of the segment before this word; list position of its first chunk, per token
      uint32_t mine[R], u_mine = 0u;
#pragma unroll
      for (int t = 0; t < R; ++t) { pos[t] = 0; mine[t] = 0u; }
      for (int w = 0; w <= w0 + warp; ++w) {
        uint32_t u = 0u;
#pragma unroll
        for (int t = 0; t < R; ++t) {
          if (t < n_tok) {
            const uint32_t routed = routed_bits(__ldg(mrow + t * dm.W + w), w, c_own);
            if (w == w0 + warp) mine[t] = routed; else pos[t] += __popc(routed);
            u |= routed;
          }
        }
        if ((c_own >> 5) == w && c_own < dm.T_a) u |= 1u << (c_own & 31);     // attended by every row
        if (w == w0 + warp) u_mine = u; else if (w >= w0) before += __popc(u);
      }
      if ((u_mine >> lane) & 1u) {
        const int c = (w0 + warp) * 32 + lane, at = before + __popc(u_mine & ((1u << lane) - 1u));
        seg_chunk[at] = c;
#pragma unroll
        for (int t = 0; t < R; ++t)
          if (t < n_tok) {
            float bv = c == c_own ? 0.f : -INFINITY;
            if (c != c_own && ((mine[t] >> lane) & 1u))
              bv = __ldg(blk_bias + (long long)grp * dm.list_rows + list_row_offset(dm, i0 + t) + pos[t] + __popc(mine[t] & ((1u << lane) - 1u)));
            seg_bias[at][t] = bv;
          }
      }
      if (warp == n_w - 1 && lane == 0) seg_n = before + __popc(u_mine);
    }
    __syncthreads();                      // (the query rows are there as well)
    const int n_items = seg_n * spc;
    for (int item = warp; item < n_items; item += NW) {
      const int at = item / spc, c = seg_chunk[at];
      const bool own = c == c_own;
      const int t_beg = c << dm.log_b, t_stop = own && dm.causal ? i0 + n_tok : min(t_beg + dm.B, dm.seq_kv);
      const int t0 = t_beg + (item - at * spc) * 32, t = t0 + my_key;
      if (t0 >= t_stop) continue;
      float s4[R][4];
#pragma unroll
      for (int rr = 0; rr < R; ++rr)
#pragma unroll
        for (int k = 0; k < 4; ++k) s4[rr][k] = 0.f;
      const T* kp[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) kp[k] = kbase + (long long)min(t0 + (lane >> 2) + 8 * k, dm.seq_kv - 1) * dm.ks[1];
      constexpr int KU = R == 4 ? 4 : 1;          // 16-element steps whose loads go out together: what the registers hold
#pragma unroll 1
      for (int d0 = 0; d0 < D; d0 += 16 * KU) {
        float4 kv[KU][4];
#pragma unroll
        for (int j = 0; j < KU; ++j)
#pragma unroll
          for (int k = 0; k < 4; ++k) kv[j][k] = load4(kp[k] + d0 + 16 * j);
#pragma unroll
        for (int j = 0; j < KU; ++j)
#pragma unroll
          for (int rr = 0; rr < R; ++rr) {
            const float4 qv = load4(&qs[rr][d0 + 16 * j + 4 * (lane & 3)]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              s4[rr][k] = fmaf(qv.x, kv[j][k].x, s4[rr][k]); s4[rr][k] = fmaf(qv.y, kv[j][k].y, s4[rr][k]);
              s4[rr][k] = fmaf(qv.z, kv[j][k].z, s4[rr][k]); s4[rr][k] = fmaf(qv.w, kv[j][k].w, s4[rr][k]);
            }
          }
      }
      // the first value rows are on their way while the probabilities are formed (R = 4)
      constexpr int VU = VPL == 4 ? 8 : 16;
      const int nt = min(32, t_stop - t0);
      const T* vp = vbase + (long long)t0 * dm.vs[1];
      float vv[VU][VPL];
      auto load_v = [&](int q0) {
#pragma unroll
        for (int u = 0; u < VU; ++u) {
          // (rows beyond the slice's end repeat its last one: probability 0)
          if constexpr (VPL == 4) {
            const float4 f = load4(vp);
            vv[u][0] = f.x; vv[u][1] = f.y; vv[u][2] = f.z; vv[u][3] = f.w;
          } else {
            const float2 f = load2(vp);
            vv[u][0] = f.x; vv[u][1] = f.y;
          }
          if (q0 + u + 1 < nt) vp += dm.vs[1];
        }
      };
      if (R == 4) load_v(0);
      float s[R], pr[R];
#pragma unroll
      for (int rr = 0; rr < R; ++rr) {
        const bool up2 = (lane & 2) != 0, up1 = (lane & 1) != 0;
        const float a0 = (up2 ? s4[rr][2] : s4[rr][0]) + __shfl_xor_sync(0xffffffffu, up2 ? s4[rr][0] : s4[rr][2], 2);
        const float a1 = (up2 ? s4[rr][3] : s4[rr][1]) + __shfl_xor_sync(0xffffffffu, up2 ? s4[rr][1] : s4[rr][3], 2);
        s[rr] = (up1 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, up1 ? a0 : a1, 1);
      }
#pragma unroll
      for (int rr = 0; rr < R; ++rr) {
        const int i = (row0 + rr) >> log_g;
        const float bv = seg_bias[at][min(i - i0, n_tok - 1)];
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
        pr[rr] = p;
      }
#pragma unroll
      for (int rr = 0; rr < R; rr += 4) store4(ps + my_key * R + rr, make_float4(pr[rr], pr[rr + 1], pr[rr + 2], pr[rr + 3]));
      __syncwarp();
#pragma unroll 1
      for (int q0 = 0; q0 < nt; q0 += VU) {
        if (R != 4 || q0 > 0) load_v(q0);
#pragma unroll
        for (int u = 0; u < VU; ++u) {
          float pq[R];
#pragma unroll
          for (int rr = 0; rr < R; rr += 4) {
            const float4 f = load4(ps + (q0 + u) * R + rr);
            pq[rr] = f.x; pq[rr + 1] = f.y; pq[rr + 2] = f.z; pq[rr + 3] = f.w;
          }
#pragma unroll
          for (int rr = 0; rr < R; ++rr)
#pragma unroll
            for (int v = 0; v < VPL; ++v) acc[rr][v] = fmaf(pq[rr], vv[u][v], acc[rr][v]);
        }
      }
      __syncwarp();
    }
  }

  // merge: every warp brings its state onto the block's maximum, the outputs are added in warp order
#pragma unroll
  for (int rr = 0; rr < R; ++rr) {
    const float ls = warp_sum(l[rr]);
    if (lane == 0) { ml[warp][rr][0] = m[rr]; ml[warp][rr][1] = ls; }
  }
  __syncthreads();                 // (and nobody reads probabilities any more)
#pragma unroll
  for (int rr = 0; rr < R; ++rr) {
    const float mq = lane < NW ? ml[lane][rr][0] : -INFINITY;
    const float M = warp_max(mq);
    const float tot = warp_sum(mq > -INFINITY ? ml[lane < NW ? lane : 0][rr][1] * __expf(mq - M) : 0.f);
    const float wgt = m[rr] > -INFINITY && tot > 0.f ? __expf(m[rr] - M) / tot : 0.f;
#pragma unroll
    for (int v = 0; v < VPL; ++v) buf[(warp * R + rr) * D + lane * VPL + v] = acc[rr][v] * wgt;
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < n_rows * D; idx += NW * 32) {
    const int rr = idx / D, k = idx % D, row = row0 + rr;
    float x = 0.f;
#pragma unroll
    for (int q = 0; q < NW; ++q) x += buf[(q * R + rr) * D + k];
    O[(long long)b * dm.os[0] + (long long)(row >> log_g) * dm.os[1] + (long long)(r * dm.g_q + (row & (dm.g_q - 1))) * dm.os[2] + k] = from_f32<T>(x);
  }
}

template <typename T, int D, int R, int NW>
static cudaError_t launch_tiles(const Dims& dm, const void* Q, const void* K, const void* V, const uint32_t* mask,
                                const float* blk_bias, void* O, cudaStream_t st) {
  const long long n_tiles = ((long long)dm.seq_q * dm.g_q + R - 1) / R;
  auto kern = attend_prefill_generic_kernel<T, D, R, NW>;
  constexpr size_t smem = buf_floats<D, R, NW>() * sizeof(float);
  static std::atomic<unsigned long long> configured{0};
  if (cudaError_t e = allow_dynamic_smem(kern, smem, configured); e != cudaSuccess) return e;
  cudaError_t e = launch_chained(kern, dim3((unsigned)(n_tiles * dm.batch * dm.h_kv)), dim3(NW * 32), smem, st, dm, (int)n_tiles,
                                 (const T*)Q, (const T*)K, (const T*)V, mask, blk_bias, (T*)O);
  count_launch();
  return e;
}

template <typename T, int D>
static cudaError_t launch_size(const Dims& dm, const void* Q, const void* K, const void* V, const uint32_t* mask,
                               const float* blk_bias, void* O, cudaStream_t st) {
  // with fewer than two eight-row tiles per SM the SMs that hold the longest tiles are what the kernel takes
  const bool few = (long long)dm.batch * dm.seq_q * dm.h_q <= 8LL * 2 * current_sm_count();
  return few ? launch_tiles<T, D, 4, 8>(dm, Q, K, V, mask, blk_bias, O, st) : launch_tiles<T, D, 8, 8>(dm, Q, K, V, mask, blk_bias, O, st);
}

cudaError_t launch_attend_prefill_generic(const Dims& dm, const void* Q, const void* K, const void* V,
                                          const uint32_t* mask, const float* blk_bias, void* O, cudaStream_t st) {
  if (dm.dtype == DASH_BF16)
    return dm.d == 128 ? launch_size<__nv_bfloat16, 128>(dm, Q, K, V, mask, blk_bias, O, st) : launch_size<__nv_bfloat16, 64>(dm, Q, K, V, mask, blk_bias, O, st);
  return dm.d == 128 ? launch_size<float, 128>(dm, Q, K, V, mask, blk_bias, O, st) : launch_size<float, 64>(dm, Q, K, V, mask, blk_bias, O, st);
}

}  // namespace dash
