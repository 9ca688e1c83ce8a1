// Stage 1 of a decode step inside a thread block (Eq. 2, Eq. 4, Algorithm 2, Proposition 1): chunk logits of one query row
// per head of a group, their entmax thresholds, and the group's routed list (used by the kernels of
// select_decode.cu and, for few groups, by the one of decode_sm100.cu).
#pragma once

#include <type_traits>

#include "common.cuh"

namespace dash {

// A sequence's length is read behind chain_wait(): the kernel before this one on the stream may be the caller's, and may be
// writing it.  Its line is brought into L2 before the wait (a prefetch reads no value: what a later read finds there is
// current), by one thread of the block; 48 paged caches take 88.8 us a step without that and 87 with.
__device__ __forceinline__ void warm_length(const int* kv_len, int b) {
  if (kv_len && threadIdx.x == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(kv_len + b));
}
__device__ __forceinline__ int sequence_length(const Dims& dm, const int* kv_len, int b) {
  return max(1, min(kv_len ? kv_len[b] : dm.seq_kv, dm.seq_kv));
}

// Sum V values held by every lane across the warp with the halving butterfly: the number of live values halves per step;
// value v ends up (fully reduced) in lane (v * 32 / V), as x[0], for V | 32.
template <int V>
__device__ __forceinline__ void warp_reduce_many(float (&x)[V], int lane) {
#pragma unroll
  for (int width = 16, live = V; width >= 1; width >>= 1) {
    if (live > 1) {
      // exchange halves: lanes with bit `width` clear keep the lower half of the live values, others the upper
      const bool upper = (lane & width) != 0;
      const int half = live / 2;
#pragma unroll
      for (int k = 0; k < V / 2; ++k) {
        if (k < half) {
          const float mine = upper ? x[k + half] : x[k];
          const float give = upper ? x[k] : x[k + half];
          x[k] = mine + __shfl_xor_sync(0xffffffffu, give, width);
        }
      }
      live = half;
    } else {
      x[0] += __shfl_xor_sync(0xffffffffu, x[0], width);
    }
  }
}

// The group's query rows, scaled.
template <typename T, int D, int G>
__device__ __forceinline__ void load_query(const Dims& dm, const T* Q, int b, int r, int lane, float (&q)[G][D / 32]) {
  constexpr int VPL = D / 32;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const T* qp = Q + (long long)b * dm.qs[0] + (long long)(r * G + g) * dm.qs[2] + lane * VPL;
#pragma unroll
    for (int v = 0; v < VPL; ++v) q[g][v] = to_f32<T>(qp[v]) * dm.x_scale;
  }
}

// Logits of candidates [c_begin, c_end), one warp per summary row, RB rows in flight per warp (warp `warp` of `n_warps`):
// store(g, c, logit).  q: the group's query rows, VPL elements per lane, scaled by x_scale; kb: the lane's share
// of summary row 0.
template <int D, int G, typename Store>
__device__ __forceinline__ void score_rows(const float (&q)[G][D / 32], const float* kb, int c_begin, int c_end, int warp, int n_warps,
                                           int lane, Store&& store) {
  constexpr int VPL = D / 32;                 // floats per lane of one summary row
  constexpr int RB = (G <= 8) ? 4 : 2;        // rows per iteration: RB * G values reduced together (<= 32)
  for (int c0 = c_begin + warp * RB; c0 < c_end; c0 += n_warps * RB) {
    float kv[RB][VPL];
#pragma unroll
    for (int u = 0; u < RB; ++u) {
      const int c = min(c0 + u, c_end - 1);
      if constexpr (VPL == 4) {
        const float4 f = __ldcs(reinterpret_cast<const float4*>(kb + (long long)c * D));   // read once: streaming
        kv[u][0] = f.x; kv[u][1] = f.y; kv[u][2] = f.z; kv[u][3] = f.w;
      } else {
        const float2 f = __ldcs(reinterpret_cast<const float2*>(kb + (long long)c * D));
        kv[u][0] = f.x; kv[u][1] = f.y;
      }
    }
    float part[RB * G];
#pragma unroll
    for (int u = 0; u < RB; ++u)
#pragma unroll
      for (int g = 0; g < G; ++g) {
        float s = 0.f;
#pragma unroll
        for (int v = 0; v < VPL; ++v) s = fmaf(q[g][v], kv[u][v], s);
        part[u * G + g] = s;
      }
    warp_reduce_many<RB * G>(part, lane);
    // value v = u*G + g is complete in lane v * (32 / (RB*G)) as part[0]
    constexpr int STRIDE = 32 / (RB * G);
    if (lane % STRIDE == 0) {
      const int v = lane / STRIDE, u = v / G, g = v % G;
      if (c0 + u < c_end) store(g, c0 + u, part[0]);
    }
  }
}

// Entmax threshold of one row of n > 0 logits in shared memory, by one warp, no barrier inside the iteration: a lane keeps
// its share of the row (RPL logits; anything beyond 32 * RPL is re-read) in registers over all passes, a pass is the
// lane's sums, two warp sums and the step.
template <int RPL>
__device__ __forceinline__ float entmax_tau(const float* x, int n_cand, int e_int, float e, int lane) {
  constexpr int MAX_NEWTON = 64, MAX_NEWTON_GENERIC = 400;
  float xr[RPL];
  float mxg = -INFINITY;
#pragma unroll
  for (int u = 0; u < RPL; ++u) {
    const int c = lane + 32 * u;
    xr[u] = c < n_cand ? x[c] : -INFINITY;
    mxg = fmaxf(mxg, xr[u]);
  }
  for (int c = lane + 32 * RPL; c < n_cand; c += 32) mxg = fmaxf(mxg, x[c]);
  mxg = warp_max(mxg);
  // moments about the maximum
  float s1 = 0.f, s2 = 0.f;
#pragma unroll
  for (int u = 0; u < RPL; ++u) {
    const float y = xr[u] > -INFINITY ? xr[u] - mxg : 0.f;
    s1 += y;
    s2 = fmaf(y, y, s2);
  }
  for (int c = lane + 32 * RPL; c < n_cand; c += 32) {
    const float y = x[c] - mxg;
    s1 += y;
    s2 = fmaf(y, y, s2);
  }
  s1 = warp_sum(s1);
  s2 = warp_sum(s2);
  float tau = mxg + entmax_start((float)n_cand, s1, s2, e_int);
  auto newton = [&](auto ei_tag) {
    constexpr int EI = decltype(ei_tag)::value;
    const int max_it = EI ? MAX_NEWTON : MAX_NEWTON_GENERIC;
    for (int it = 0; it < max_it; ++it) {
      float F[4] = {0.f, 0.f, 0.f, 0.f}, Gs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int u = 0; u < RPL; ++u) {
        const float m = fmaxf(xr[u] - tau, 0.f);
        F[u & 3] += pow_e(m, EI, e);
        Gs[u & 3] += pow_em1(m, EI, e);
      }
      for (int c = lane + 32 * RPL; c < n_cand; c += 32) {
        const float m = fmaxf(x[c] - tau, 0.f);
        F[0] += pow_e(m, EI, e);
        Gs[0] += pow_em1(m, EI, e);
      }
      const float f = warp_sum((F[0] + F[1]) + (F[2] + F[3]));
      const float gs = warp_sum((Gs[0] + Gs[1]) + (Gs[2] + Gs[3]));
      const float nt = newton_next(tau, f, gs, EI, e);
      if (nt == tau) break;
      tau = nt;
      if (newton_settled(f, gs, (float)n_cand, EI)) break;
    }
  };
  switch (e_int) {
    case 1: newton(std::integral_constant<int, 1>{}); break;
    case 2: newton(std::integral_constant<int, 2>{}); break;
    case 4: newton(std::integral_constant<int, 4>{}); break;
    default: newton(std::integral_constant<int, 0>{}); break;
  }
  return tau;
}

// Pitch (floats) of a row of n logits in shared memory.
__host__ __device__ inline int route_stride(int n) { return ((n + 31) / 32) * 32 + 32; }

// Routes one group: X [G][stride] holds the logits of its n_cand candidates (synchronised), n_vis - n_cand window chunks
// follow them.  Called by every thread of a block of NW warps.  set_word(j, word) is called once per mask word, listed(n)
// by every thread once the list's length is known, emit(pos, chunk, bias) once per list entry.  MAXR: logits per lane
// that a Newton warp may keep in registers.  taus: G floats; wsum: n_words floats; wcnt: n_words + 1 ints.
template <int G, int NW, int MAXR, typename SetWord, typename Listed, typename Emit>
__device__ __forceinline__ void route_group(const Dims& dm, float* X, int stride, int n_cand, int n_vis, int n_words, float* taus,
                                            float* wsum, int* wcnt, int warp, int lane, SetWord&& set_word, Listed&& listed, Emit&& emit) {
  const int e_int = dm.e_int;
  const float e = dm.e;
  for (int g = warp; g < G; g += NW) {
    const float* x = X + (size_t)g * stride;
    float tau = 0.f;
    // (a pass costs its RPL terms whether the row has them or not)
    if (MAXR >= 64 && n_cand > 512) tau = entmax_tau<(MAXR >= 64 ? 64 : 16)>(x, n_cand, e_int, e, lane);
    else if (n_cand > 128) tau = entmax_tau<16>(x, n_cand, e_int, e, lane);
    else if (n_cand > 0) tau = entmax_tau<4>(x, n_cand, e_int, e, lane);
    if (lane == 0) taus[g] = tau;
  }
  __syncthreads();
  // pass 1: one warp per 32-chunk mask word: support bits, log w (stashed over head 0's logits)
  const float log_gq = logf((float)G);
  for (int j = warp; j < n_words; j += NW) {
    const int c = j * 32 + lane;
    bool sel = false;
    float lw = INFINITY;
    if (c < n_cand) {
      float mg[G], mstar = 0.f;
#pragma unroll
      for (int g = 0; g < G; ++g) {
        mg[g] = X[(size_t)g * stride + c] - taus[g];
        mstar = fmaxf(mstar, mg[g]);
      }
      if (mstar > 0.f) {
        sel = true;
        const float inv = 1.f / mstar;
        float s = 0.f;
#pragma unroll
        for (int g = 0; g < G; ++g) s += pow_e(fmaxf(mg[g], 0.f) * inv, e_int, e);
        lw = e * logf(mstar) + logf(s) - log_gq;
      }
    }
    const float ls = warp_sum(sel ? lw : 0.f);
    if (c >= n_cand && c < n_vis) {                 // window chunk: listed with bias 0, outside mu
      sel = true;
      lw = -INFINITY;
    }
    const uint32_t word = __ballot_sync(0xffffffffu, sel);
    if (c < n_vis) X[c] = lw;                       // +inf marks "not routed", -inf a window chunk
    if (lane == 0) {
      set_word(j, word);
      wsum[j] = ls;
      wcnt[j] = __popc(word);
    }
  }
  __syncthreads();
  // exclusive prefix of the per-word counts and the total of log w: every warp for itself where one round of lanes covers
  // the words, else warp 0 for all
  float tot = 0.f;
  int before = 0, nlist;
  if (n_words <= 32) {
    const int v = lane < n_words ? wcnt[lane] : 0;
    tot = warp_sum(lane < n_words ? wsum[lane] : 0.f);
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    nlist = __shfl_sync(0xffffffffu, incl, 31);
    before = incl - v;
  } else {
    if (warp == 0) {
      int base = 0;
      for (int j0 = 0; j0 < n_words; j0 += 32) {
        const int j = j0 + lane;
        const int v = j < n_words ? wcnt[j] : 0;
        const float sv = j < n_words ? wsum[j] : 0.f;
        int incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += t;
        }
        if (j < n_words) wcnt[j] = base + incl - v;
        base += __shfl_sync(0xffffffffu, incl, 31);
        tot += warp_sum(sv);
      }
      __syncwarp();
      if (lane == 0) {
        wcnt[n_words] = base;
        wsum[0] = tot;
      }
    }
    __syncthreads();
    nlist = wcnt[n_words];
    tot = wsum[0];
  }
  const int nsel = nlist - (n_vis - n_cand);     // routed only: the denominator of mu
  const float mu = nsel > 0 ? tot / (float)nsel : 0.f;
  listed(nlist);
  for (int j = warp; j * 32 < n_vis; j += NW) {
    const int c = j * 32 + lane;
    const float lw = (c < n_vis) ? X[c] : INFINITY;
    const bool sel = lw < INFINITY;
    const uint32_t word = __ballot_sync(0xffffffffu, sel);
    const int base = n_words <= 32 ? __shfl_sync(0xffffffffu, before, j & 31) : wcnt[j];
    if (sel) emit(base + __popc(word & ((1u << lane) - 1u)), c, lw == -INFINITY ? 0.f : (lw - mu) * dm.inv_sigma);
  }
}

}  // namespace dash
