// The walk of a query tile over the union of its rows' routed chunks, as the producer warps of the tensor-core prefill
// kernels (forward, dQ) make it: one warp, lane t looking after the tokens t, t + 32, ... of the tile.
#pragma once

#include "common.cuh"

namespace dash {

// A token's routed chunks in mask word w: its own chunk c (whose bit is set in every row) and later ones cleared.
__device__ __forceinline__ uint32_t routed_bits(uint32_t word, int w, int c) {
  return w < (c >> 5) ? word : w == (c >> 5) ? word & ((1u << (c & 31)) - 1u) : 0u;
}

// CPS: chunks per 64-token step.  WIDE: the tile's tokens may have different own chunks.  TPL: tokens per lane.
template <int CPS, bool WIDE, int TPL>
struct TileWalk {
  const uint32_t* rows;      // mask words of the tile's first token
  int W, n_live, lane;       // words per row; tokens of the tile inside the sequence
  int c_first, n_words;      // own chunk of the tile's first token; mask words that can hold a routed chunk
  int co[WIDE ? TPL : 1];    // own chunks of this lane's tokens
  uint32_t rw[TPL], rw_n[TPL];   // routed bits of the word being walked, and the raw next word
  int seen[TPL];             // routed chunks of this lane's tokens in the words already walked
  uint32_t u;
  int w;

  __device__ __forceinline__ int own(int q) const { return WIDE ? co[WIDE ? q : 0] : c_first; }
  __device__ __forceinline__ TileWalk(const Dims& dm, const uint32_t* mask, long long row0, int i0, int TQ, int lane_) {
    W = dm.W;
    lane = lane_;
    rows = mask + (row0 + i0) * dm.W;
    n_live = min(TQ, dm.seq_q - i0);
    c_first = i0 >> dm.log_b;
    n_words = ((WIDE ? (i0 + n_live - 1) >> dm.log_b : c_first) >> 5) + 1;
    if constexpr (WIDE) {
#pragma unroll
      for (int q = 0; q < TPL; ++q) co[q] = (i0 + lane + 32 * q) >> dm.log_b;
    }
  }
  // Number of chunks in the union.  Four mask words per sweep: a lane's loads are in flight together (one L2 round trip
  // per four words instead of one per word; the issuing threads wait for this count before their second step).
  __device__ __forceinline__ int count() const {
    int total = 0;
    for (int w0 = 0; w0 < n_words; w0 += 4) {
      uint32_t uu[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int q = 0; q < TPL; ++q) {
        const int t = lane + 32 * q;
        if (t < n_live) {
          const uint32_t* mp = rows + (long long)t * W + w0;
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (w0 + k < n_words) uu[k] |= WIDE ? routed_bits(mp[k], w0 + k, own(q)) : mp[k];
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (w0 + k < n_words) {
          const uint32_t v = __reduce_or_sync(0xffffffffu, uu[k]);
          total += __popc(WIDE ? v : routed_bits(v, w0 + k, c_first));
        }
      }
    }
    return total;
  }
  __device__ __forceinline__ void load(int word) {
#pragma unroll
    for (int q = 0; q < TPL; ++q) {
      const int t = lane + 32 * q;
      rw_n[q] = t < n_live ? rows[(long long)t * W + word] : 0u;
    }
  }
  __device__ __forceinline__ void take() {     // the loaded word becomes the walked one
    u = 0u;
#pragma unroll
    for (int q = 0; q < TPL; ++q) {
      rw[q] = routed_bits(rw_n[q], w, own(q));
      u |= rw[q];
    }
    u = __reduce_or_sync(0xffffffffu, u);
    if (w + 1 < n_words) load(w + 1);
  }
  __device__ __forceinline__ void start() {
    w = 0;
#pragma unroll
    for (int q = 0; q < TPL; ++q) seen[q] = 0;
    load(0);
    take();
  }
  // The next chunks of the union, ascending, at most CPS of them: returns their number m and, for each, the position of
  // the chunk in the lists of this lane's tokens (-1: the token did not route it).  A position is the count of the
  // token's routed bits below the chunk, so nothing walks the lists entry by entry.
  // (POS = false: chunks only.)
  template <bool POS = true>
  __device__ __forceinline__ int next(int (&cs)[CPS], int (&pos)[CPS][TPL]) {
    int m = 0;
#pragma unroll
    for (int s = 0; s < CPS; ++s) {
      while (u == 0u && w < n_words) {
        if constexpr (POS) {
#pragma unroll
          for (int q = 0; q < TPL; ++q) seen[q] += __popc(rw[q]);
        }
        if (++w < n_words) take();
      }
      const bool got = u != 0u;
      const int bit = got ? __ffs(u) - 1 : 0;
      u &= u - 1;                               // (0 stays 0)
      if (got) {
        cs[s] = w * 32 + bit;
        ++m;
      } else {
        cs[s] = s > 0 ? cs[s > 0 ? s - 1 : 0] : 0;      // a short last step repeats its last chunk
      }
#pragma unroll
      for (int q = 0; q < TPL; ++q)
        if constexpr (POS) pos[s][q] = got && ((rw[q] >> bit) & 1u) ? seen[q] + __popc(rw[q] & ((1u << bit) - 1u)) : -1;
    }
    return m;
  }
};

}  // namespace dash
