// What the tensor-core kernels of the Stage-2 backward share (prefill_bwd_sm100.cu, prefill_bwd_stats_sm100.cu).
#pragma once
#include <cuda.h>

#include "common.cuh"
#include "sm100_ptx.cuh"
#include "tile_walk.cuh"

namespace dash {

constexpr int BWD_NKV = 64;                 // keys per step / per slice
constexpr float LOG2E = 1.4426950408889634f;

struct BwdArgs {
  Dims dm;
  int TQ;             // tokens per query tile
  int n_tiles;        // query tiles per (batch, KV head)
  int n_slices;       // 64-key slices per (batch, KV head)
  int n_split;        // blocks that share a slice's query tiles (1: they write dK / dV, more: they add to them)
  int inject;         // test hook: 1 = the statistics pass never loads the own chunk's keys (the waits for them run out)
  long long wait_limit;
  const __nv_bfloat16* Q;
  const __nv_bfloat16* dO;
  const uint32_t* mask;
  const float* blk_bias;
  RowStats stats;
  int* marks;         // counts, in the layout of the lists
  __nv_bfloat16* dQ;
  float* dK;
  float* dV;
  float* dbias;
  StatusBlock* sb;
};

struct BwdMaps {
  CUtensorMap q, g, qr, gr, k, v, kc, vc;      // q, g: a query tile per box; qr, gr: a run of at most 32 tokens; kc, vc: one chunk per box (query-tile-stationary kernels pack chunks below 64 tokens)
};

cudaError_t launch_attend_bwd_stats(const BwdArgs& a, const BwdMaps& m, cudaStream_t st);

// What a query-tile-stationary kernel's threads need to know of a step's columns, beside the K / V tiles: a ring of MD steps.
// POS: also the chunk's position in the token's list (-1: own chunk or not routed).
template <int CPS, int MTQ, int MD, bool POS>
struct StepMeta {
  int kvbase[MD][CPS];
  float bias[MD][CPS][MTQ];
  int pos[POS ? MD : 1][POS ? CPS : 1][POS ? MTQ : 1];
};

// Warps of the query-tile-stationary kernels: three warpgroups that take the steps in turn (a thread = a tile row), and one of
// service warps.  A step costs a thread some 600 clocks of barrier tests, tensor-memory loads and arrivals whatever its
// width, so a warpgroup takes whole steps, every third one, instead of a share of every step.  Tiles and records come from two
// warps: one that does both needs 900 clocks a step, more than the products take.
constexpr int BWD_ROW_WG = 3, BWD_ROW_THREADS = (BWD_ROW_WG + 1) * 128, BWD_W_TILES = 12, BWD_W_RECORDS = 13, BWD_W_SD = 14, BWD_W_DQ = 15;
// Registers per thread after the re-division (128 each at launch): a producer lane of a wide tile looks after more tokens.
__host__ __device__ constexpr int bwd_regs_service(int wt, int cps) { return wt > 2 || (wt > 0 && cps > 2) ? 104 : wt > 0 || cps > 1 ? 80 : 56; }
__host__ __device__ constexpr int bwd_regs_row(int wt, int cps) { return (4 * 128 - bwd_regs_service(wt, cps)) / 3 / 8 * 8; }

// 4 or 16 bytes global -> shared, asynchronously; the barrier gets one arrival once this thread's copies have landed.
__device__ __forceinline__ void copy_async4(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void arrive_after_copies(uint32_t bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}

// A ring position that is stepped instead of divided: index (below N) and phase parity of step j.
template <int N>
struct RingPos {
  int at = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ void step() {
    if (++at == N) {
      at = 0;
      phase ^= 1u;
    }
  }
};

// The forward kernel's walk (own chunks, then the union of the tile's routed chunks, 64 tokens per step), made by two warps:
// with TILES one fills a ring of DK K tiles and one of DV V tiles, without it the other a ring of DK step records.  Step j's
// barrier is full[j mod DK], with one arrival: of the tiles with the byte count of both.
// `free_for(j)` waits until step j's tiles and record may be overwritten (called for j >= min(DK, DV)); `publish(n)` is
// told the number of steps.  A walk that was cut short (a wait ran out) lets its copies in flight land (bounded).
template <int HD, int CPS, int WT, int DK, int DV, bool TILES, bool POS, typename Meta, typename FreeFor, typename Publish>
__device__ __forceinline__ void produce_steps(const BwdArgs& a, const CUtensorMap* tmK, const CUtensorMap* tmV, int grp, int i0, int lane,
                                              uint32_t ring_k, uint32_t ring_v, const unsigned long long* full, Meta* meta,
                                              bool skip_own_k, FreeFor&& free_for, Publish&& publish) {
  constexpr bool WIDE = WT > 0;
  constexpr int TPL = WIDE ? WT : 2, NKV = BWD_NKV, W = NKV / CPS;
  constexpr uint32_t TILE_BYTES = NKV * HD * 2;
  const Dims& dm = a.dm;
  const int TQ = a.TQ, b = grp / dm.h_kv, r = grp % dm.h_kv;
  const int c_own = i0 >> dm.log_b, sub_per_blk = dm.B / NKV;
  const int own_steps = WIDE ? (TQ + NKV - 1) / NKV : (i0 % dm.B) / NKV + 1;      // at most 2
  RingPos<DK> pk;
  RingPos<DV> pv;
  auto bar_of = [&](int at) { return ptx::smem_u32(full + at); };
  // (by the whole warp: an elected lane issues, so that the operands are uniform; sixteen copies a step of chunks of 16 tokens)
  auto load = [&](const int* kvs, bool with_k) {
    int at[CPS];
#pragma unroll
    for (int s = 0; s < CPS; ++s) at[s] = __shfl_sync(0xffffffffu, kvs[s], 0);
    if (ptx::elect_one()) {
      const uint32_t bar = bar_of(pk.at);
      ptx::mbar_arrive_expect_tx(bar, 2 * TILE_BYTES);
#pragma unroll
      for (int s = 0; s < CPS; ++s) {
        const uint32_t k = ring_k + pk.at * TILE_BYTES + s * W * 128, v = ring_v + pv.at * TILE_BYTES + s * W * 128;
        if (with_k) {
          ptx::tma_load_4d(k, tmK, bar, 0, r, at[s], b);
          if constexpr (HD == 128) ptx::tma_load_4d(k + TILE_BYTES / 2, tmK, bar, 64, r, at[s], b);
        }
        ptx::tma_load_4d(v, tmV, bar, 0, r, at[s], b);
        if constexpr (HD == 128) ptx::tma_load_4d(v + TILE_BYTES / 2, tmV, bar, 64, r, at[s], b);
      }
    }
    __syncwarp();
  };
  auto record_done = [&]() {
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(bar_of(pk.at));
  };
  // own chunks first: their tiles need nothing from the mask
  for (int sub = 0; sub < own_steps; ++sub) {
    int kvs[CPS];
    const int kv0 = WIDE ? i0 + sub * NKV : c_own * dm.B + sub * NKV;
#pragma unroll
    for (int s = 0; s < CPS; ++s) kvs[s] = WIDE && kv0 + s * W < i0 + TQ ? kv0 + s * W : kv0;
    if constexpr (TILES) {
      load(kvs, !skip_own_k);
    } else {
      for (int t = lane; t < TQ; t += 32)
#pragma unroll
        for (int s = 0; s < CPS; ++s) {
          meta->bias[sub][s][t] = (WIDE ? (kv0 + s * W) >> dm.log_b == (i0 + t) >> dm.log_b : s == 0) ? 0.f : -INFINITY;
          if constexpr (POS) meta->pos[sub][s][t] = -1;
        }
#pragma unroll
      for (int s = 0; s < CPS; ++s)
        if (lane == s) meta->kvbase[sub][s] = kvs[s];
      record_done();
    }
    pk.step();
    pv.step();
  }
  TileWalk<CPS, WIDE, TPL> walk(dm, a.mask, (long long)grp * dm.seq_q, i0, TQ, lane);
  const int total = walk.count();
  const int n_steps = (CPS > 1 ? (total + CPS - 1) / CPS : total * sub_per_blk) + own_steps;
  publish(n_steps);
  walk.start();
  bool ok = true;
  int j = own_steps;
  if constexpr (TILES) {
    while (j < n_steps && ok) {
      int cs[CPS], pos[CPS][TPL];
      walk.template next<false>(cs, pos);
      for (int sub = 0; sub < (CPS > 1 ? 1 : sub_per_blk); ++sub) {
        int kvs[CPS];
#pragma unroll
        for (int s = 0; s < CPS; ++s) kvs[s] = cs[s] * dm.B + sub * NKV;
        if (j >= (DK < DV ? DK : DV)) ok = free_for(j);
        if (!ok) break;
        load(kvs, true);
        pk.step();
        pv.step();
        ++j;
      }
    }
  } else {
    const float* list[TPL];
#pragma unroll
    for (int q = 0; q < TPL; ++q)
      list[q] = a.blk_bias + (long long)grp * dm.list_rows + list_row_offset(dm, min(i0 + lane + 32 * q, dm.seq_q - 1));
    // A chunk's biases are asked for before the step before is handed on, and stored when its own turn comes.  (Loads: a warp's 32 list
    // entries lie in 32 places, and an asynchronous copy of them holds the warp up for some 200 clk, sixteen of them a step in
    // chunks of 16 with 128 tokens, 6000 clk a step.)
    int cs[CPS], pos[CPS][TPL];
    float bias[CPS][TPL];
    auto ask = [&]() {
      walk.next(cs, pos);
#pragma unroll
      for (int s = 0; s < CPS; ++s)
#pragma unroll
        for (int q = 0; q < TPL; ++q) {
          bias[s][q] = -INFINITY;
          if (pos[s][q] >= 0) bias[s][q] = __ldg(list[q] + pos[s][q]);
        }
    };
    if (j < n_steps) ask();
    while (j < n_steps && ok) {
      for (int sub = 0; sub < (CPS > 1 ? 1 : sub_per_blk); ++sub) {
        if (j >= DK) ok = free_for(j);
        if (!ok) break;
        const int ms = pk.at;
#pragma unroll
        for (int s = 0; s < CPS; ++s) {
#pragma unroll
          for (int q = 0; q < TPL; ++q) {
            const int t = lane + 32 * q;
            if (t < TQ) {
              meta->bias[ms][s][t] = bias[s][q];
              if constexpr (POS) meta->pos[ms][s][t] = pos[s][q];
            }
          }
          if (lane == s) meta->kvbase[ms][s] = cs[s] * dm.B + sub * NKV;
        }
        record_done();
        pk.step();
        ++j;
      }
      if (j < n_steps && ok) ask();
    }
  }
  if (TILES && !ok && lane == 0) {
    for (int last = j - 1; last >= (skip_own_k ? own_steps : 0) && last > j - 1 - DK; --last)
      for (int k = 0; k < 200000 && !ptx::mbar_try_wait(bar_of(last % DK), (uint32_t)(last / DK) & 1u); ++k) {}
  }
}

}  // namespace dash
