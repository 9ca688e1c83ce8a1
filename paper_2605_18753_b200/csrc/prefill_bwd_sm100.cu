// Stage 2 backward, prefill, tensor-core path for sm_100a (Section 3.5: the backward pass reuses the forward pass's bit
// mask; Eq. 7 in the form of Proposition 1 is what is differentiated, with the routing held fixed).
//
// With P = softmax of the row's logits l_j = <q,k_j>/sqrt(d) + bias_c(j) over its selected tokens, dP = dO V^T,
// delta = <O, dO> per row and dS = P o (dP - delta):
//     dQ = dS K / sqrt(d),   dK = dS^T Q / sqrt(d),   dV = P^T dO,   dbias_c = sum of dS over the chunk's tokens.
// Three launches behind the statistics pass (prefill_bwd_stats_sm100.cu; it leaves the log-sum-exp and delta of every row):
//   list_marks_kernel       per row, the number of routed chunks in the mask words before each word (so that a row's
//                           list entry for a chunk can be found from one word of its mask);
//   attend_bwd_dkv_kernel   key-slice stationary (64 keys of one KV head): gathers the tokens that attend the slice (those of
//                           its own chunks, causally masked, then every later one that routed one of its chunks) into steps
//                           of 128 (token, head) rows, computes S and dP, and accumulates dV^T += dO^T P and dK^T += Q^T dS
//                           in tensor memory (P and dS pass through shared memory as bf16 MN-major operands);
//   attend_bwd_dq_kernel    query-tile stationary, the forward kernel's walk over the union of the tile's routed
//                           chunks: S = Q K^T and dP = dO V^T into tensor memory, dS (bf16) back into tensor memory,
//                           dQ += dS K accumulated in tensor memory; dbias from the row sums of dS.
// What passes between them needs no scratch of its own: a row's statistics sit in the first eight bytes of its dQ row until
// the dQ kernel, which owns the row, overwrites them; the counts sit in the rows' regions of dbias (a row with own chunk c has
// c entries there, and c >= floor(c / 32)), which the dQ kernel's block zeroes for its own rows first.
// A block whose wait ran out writes NaN in the place of its statistics or gradients: the entry point without a status word has
// no other way to say so, and what the buffers held as scratch must not pass for gradients.
//
// bf16 operands, fp32 accumulation.  P2 instantiations (the entry point that takes every shape, which computed P and dS in
// fp32 when it ran on CUDA cores) carry P and dS as two bf16 terms (hi + lo, 16 bits of mantissa) through every product;
// the others round them to bf16.  Tiles as in the forward kernel (prefill_sm100.cu).  Every wait is bounded.
//
// Bound by the chain of a step (tile landed -> S, dP -> P, dS -> accumulating products), one block per SM.  2 x 1500 tokens,
// 8/2 heads, d 64, chunks of 32: 2.02 ms on CUDA cores (one warp per row and head, two vector reductions per token and
// row) -> 0.11 ms; 8192 tokens, 32/8 heads, d 128, chunks of 64, one term: statistics 0.33, dK / dV 0.56, dQ 0.51 ms.
#include <cuda.h>

#include <algorithm>

#include "bwd_sm100.cuh"
#include "tensor_map.cuh"

namespace dash {

namespace {

constexpr int NKV = BWD_NKV;

// Where a row's counts start (entry w - 1: routed chunks in mask words 0 .. w - 1).
__device__ __forceinline__ long long marks_of(const Dims& dm, long long grp, int i) {
  return grp * dm.list_rows + list_row_offset(dm, i);
}

__global__ void __launch_bounds__(256)
list_marks_kernel(Dims dm, const uint32_t* __restrict__ mask, int* __restrict__ marks, float* zero_a, float* zero_b, long long zero_n) {
  chain_wait();
  chain_release();
  const long long thread = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (zero_n > 0) {            // dK, dV: several blocks of the next kernel add to them
    zero_floats(zero_a, zero_n, thread, (long long)gridDim.x * blockDim.x);
    zero_floats(zero_b, zero_n, thread, (long long)gridDim.x * blockDim.x);
  }
  if (thread >= (long long)dm.batch * dm.h_kv * dm.seq_q) return;
  const long long grp = thread / dm.seq_q;
  const int i = (int)(thread % dm.seq_q), last_w = (i >> dm.log_b) >> 5;      // (the words before the own chunk's hold routed chunks only)
  const uint32_t* row = mask + thread * dm.W;
  int* out = marks + marks_of(dm, grp, i);
  int acc = 0;
  for (int w0 = 0; w0 < last_w; w0 += 4) {
    uint32_t word[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) word[k] = w0 + k < last_w ? row[w0 + k] : 0u;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      acc += __popc(word[k]);
      if (w0 + k < last_w) out[w0 + k] = acc;
    }
  }
}

// P or dS of 32 columns as packed bf16 pairs; with P2 also the remainders (x = hi + lo)
template <bool P2>
__device__ __forceinline__ void pack_terms(const float (&x)[32], uint32_t (&hi)[16], uint32_t (&lo)[16]) {
#pragma unroll
  for (int c = 0; c < 32; c += 2) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x[c], x[c + 1]);
    hi[c >> 1] = *reinterpret_cast<const uint32_t*>(&h);
    if constexpr (P2) {
      const float2 hf = __bfloat1622float2(h);
      const __nv_bfloat162 l = __floats2bfloat162_rn(x[c] - hf.x, x[c + 1] - hf.y);
      lo[c >> 1] = *reinterpret_cast<const uint32_t*>(&l);
    }
  }
}

// ===================================================================================================================
// dQ and dbias: query-tile stationary
// ===================================================================================================================
namespace dq {

// Warps as in the statistics pass (bwd_sm100.cuh): three warpgroups form dS, taking the steps in turn.  A V tile is free when its dP product is done, a K tile and a step record when the step's dQ product is:
// rings of their own, so that a step's tiles have landed by the time its S / dP slot is free.
constexpr int THREADS = BWD_ROW_THREADS;
constexpr int KST = 5, VST = 3;         // ring of K tiles and step records; ring of V tiles and of S / dP slots
constexpr uint32_t TMEM_COLS = 512;     // S [0,192) dP [192,384) dQ [384,512)
constexpr uint32_t COL_DP = 192, COL_DQ = 384;
enum Bar { QD_FULL = 0, META_READY, SD_FULL = 2, DS_FULL = 5, KV_FULL = 8, K_FREE = 13, REC_FULL = 18, N_BARS = 23 };
template <int CPS, int MTQ>
struct MiscT {
  unsigned long long bar[N_BARS];
  uint32_t tmem_base;
  int n_steps;
  int abort_flag;
  StepMeta<CPS, MTQ, KST, true> meta;
};
template <int HD, int CPS, int MTQ>
struct Layout {
  static constexpr uint32_t Q_BYTES = 128 * HD * 2;          // HD = 128: 32 KiB, two 128x64 regions
  static constexpr uint32_t KV_TILE_BYTES = NKV * HD * 2;
  static constexpr uint32_t OFF_Q = 0, OFF_DO = OFF_Q + Q_BYTES, OFF_K = OFF_DO + Q_BYTES, OFF_V = OFF_K + KST * KV_TILE_BYTES,
                            OFF_MISC = OFF_V + VST * KV_TILE_BYTES, SMEM = OFF_MISC + sizeof(MiscT<CPS, MTQ>);
  static_assert(SMEM <= 232448, "one block per SM");
};

template <int HD, int CPS, int WT, bool P2>
__global__ void __launch_bounds__(THREADS, 1)
attend_bwd_dq_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmDO,
                     const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, BwdArgs a) {
  constexpr int MTQ = 32 * (WT > 0 ? WT : 2), W = NKV / CPS;
  using LY = Layout<HD, CPS, MTQ>;
  using Misc = MiscT<CPS, MTQ>;
  constexpr uint32_t Q_BYTES = LY::Q_BYTES, KV_TILE_BYTES = LY::KV_TILE_BYTES, OFF_Q = LY::OFF_Q, OFF_DO = LY::OFF_DO,
                     OFF_K = LY::OFF_K, OFF_V = LY::OFF_V;
  extern __shared__ __align__(1024) uint8_t smem[];
  Misc* misc = reinterpret_cast<Misc*>(smem + LY::OFF_MISC);
  const Dims& dm = a.dm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t sbase = ptx::smem_u32(smem);
  auto bar = [&](int i) { return ptx::smem_u32(&misc->bar[i]); };
  volatile int* abort_flag = &misc->abort_flag;
  const long long wait_limit = a.wait_limit;
  auto wait_all = [&](uint32_t barrier, uint32_t parity) { return ptx::mbar_wait_warp(barrier, parity, abort_flag, wait_limit); };

  const int groups = dm.batch * dm.h_kv;
  const int tile = a.n_tiles - 1 - (int)(blockIdx.x / groups);  // late (long) tiles first
  const int grp = (int)(blockIdx.x % groups);
  const int b = grp / dm.h_kv, r = grp % dm.h_kv;
  const int TQ = a.TQ, g_q = dm.g_q;
  const int i0 = tile * TQ;

  if (tid == 0) {
    misc->abort_flag = ((sbase & 1023u) != 0u) ? 1 : 0;
    if (misc->abort_flag) report_error(a.sb, DASH_ERR_CUDA, 110);
    ptx::mbar_init(bar(QD_FULL), 1);
    ptx::mbar_init(bar(META_READY), 1);
    for (int s = 0; s < VST; ++s) {
      ptx::mbar_init(bar(SD_FULL + s), 1);
      ptx::mbar_init(bar(DS_FULL + s), 128);
    }
    for (int s = 0; s < KST; ++s) {
      ptx::mbar_init(bar(KV_FULL + s), 1);
      ptx::mbar_init(bar(REC_FULL + s), 1);
      ptx::mbar_init(bar(K_FREE + s), 1);
    }
    ptx::fence_barrier_init();
  }
  if (warp == BWD_W_SD) {
    ptx::tmem_alloc(ptx::smem_u32(&misc->tmem_base), TMEM_COLS);
    ptx::tmem_relinquish();
    ptx::tc_fence_before();
  }
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = misc->tmem_base;
  chain_wait();
  chain_release();
  {
    // this tile's rows' list regions follow each other: their dbias starts from zero (the marks have been read)
    const long long at = (long long)grp * dm.list_rows, lo = list_row_offset(dm, i0),
                    hi = i0 + TQ < dm.seq_q ? list_row_offset(dm, i0 + TQ) : dm.list_rows;
    for (long long k = lo + tid; k < hi; k += THREADS) a.dbias[at + k] = 0.f;
  }
  if (a.sb && *reinterpret_cast<volatile int*>(&a.sb->status) != 0) *abort_flag = 1;
  __syncthreads();

  if (warp >= BWD_W_TILES) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(bwd_regs_service(WT, CPS)));
  if (warp == BWD_W_TILES) {
    if (lane == 0) {
      ptx::prefetch_tensormap(&tmQ);
      ptx::prefetch_tensormap(&tmDO);
      ptx::prefetch_tensormap(&tmK);
      ptx::prefetch_tensormap(&tmV);
      ptx::mbar_arrive_expect_tx(bar(QD_FULL), 2 * Q_BYTES);
      ptx::tma_load_4d(sbase + OFF_Q, &tmQ, bar(QD_FULL), 0, r * g_q, i0, b);
      if constexpr (HD == 128) ptx::tma_load_4d(sbase + OFF_Q + Q_BYTES / 2, &tmQ, bar(QD_FULL), 64, r * g_q, i0, b);
      ptx::tma_load_4d(sbase + OFF_DO, &tmDO, bar(QD_FULL), 0, r * g_q, i0, b);
      if constexpr (HD == 128) ptx::tma_load_4d(sbase + OFF_DO + Q_BYTES / 2, &tmDO, bar(QD_FULL), 64, r * g_q, i0, b);
    }
    produce_steps<HD, CPS, WT, KST, VST, true, true>(
        a, &tmK, &tmV, grp, i0, lane, sbase + OFF_K, sbase + OFF_V, &misc->bar[KV_FULL], &misc->meta, false,
        [&](int j) {
          return wait_all(bar(SD_FULL + j % VST), (uint32_t)(j / VST - 1) & 1u) &&
                 (j < KST || wait_all(bar(K_FREE + j % KST), (uint32_t)(j / KST - 1) & 1u));
        },
        [&](int n) {
          if (lane == 0) {
            misc->n_steps = n;
            ptx::mbar_arrive(bar(META_READY));
          }
        });
    if (lane == 0 && *abort_flag)
      for (int k = 0; k < 200000 && !ptx::mbar_try_wait(bar(QD_FULL), 0); ++k) {}
  } else if (warp == BWD_W_RECORDS) {
    produce_steps<HD, CPS, WT, KST, VST, false, true>(
        a, &tmK, &tmV, grp, i0, lane, 0u, 0u, &misc->bar[REC_FULL], &misc->meta, false,
        [&](int j) { return j < KST || wait_all(bar(K_FREE + j % KST), (uint32_t)(j / KST - 1) & 1u); }, [](int) {});
  } else if (warp == BWD_W_SD) {
    // =========================== issuer of S = Q K^T and dP = dO V^T ===========================
    // Slot j mod 3 of S / dP is free once the dQ product of step j-3 is done (which reads dS from it).
    bool ok = wait_all(bar(QD_FULL), 0);
    int n_steps = 0x7fffffff;            // known from step 1 on; step 0 (the own chunk) always exists
    constexpr uint32_t IDESC_S = ptx::idesc_bf16_f32(128, NKV, false, false);
    const uint64_t qd = ptx::smem_desc_sw128(sbase + OFF_Q, 16, 1024), gd = ptx::smem_desc_sw128(sbase + OFF_DO, 16, 1024);
    const uint64_t kd0 = ptx::smem_desc_sw128(sbase + OFF_K, 16, 1024), vd0 = ptx::smem_desc_sw128(sbase + OFF_V, 16, 1024);
    const uint32_t d0 = __shfl_sync(0xffffffffu, tmem, 0);
    RingPos<KST> pk, pf;                 // step j's K tile; step j-3's, whose release frees the slot
    RingPos<VST> pv;
    for (int j = 0; j < n_steps && ok; ++j, pk.step(), pv.step()) {
      if (j == 1) {
        ok = wait_all(bar(META_READY), 0);
        if (!ok) break;
        n_steps = __shfl_sync(0xffffffffu, misc->n_steps, 0);
        if (j >= n_steps) break;
      }
      ok = wait_all(bar(KV_FULL + pk.at), pk.phase);
      if (ok && j >= VST) {
        ok = wait_all(bar(K_FREE + pf.at), pf.phase);
        pf.step();
      }
      if (!ok) break;
      ptx::tc_fence_after();
      const uint64_t ktile = (uint64_t)((pk.at * KV_TILE_BYTES) >> 4), vtile = (uint64_t)((pv.at * KV_TILE_BYTES) >> 4);
      if (ptx::elect_one()) {
#pragma unroll
        for (int k = 0; k < HD / 16; ++k) {
          const uint64_t off_a = (uint64_t)(((k >> 2) * (Q_BYTES / 2) + (k & 3) * 32) >> 4);
          const uint64_t off_b = (uint64_t)(((k >> 2) * (KV_TILE_BYTES / 2) + (k & 3) * 32) >> 4);
          ptx::mma_bf16_ss(d0 + pv.at * NKV, qd + off_a, kd0 + ktile + off_b, IDESC_S, k > 0 ? 1u : 0u);
        }
#pragma unroll
        for (int k = 0; k < HD / 16; ++k) {
          const uint64_t off_a = (uint64_t)(((k >> 2) * (Q_BYTES / 2) + (k & 3) * 32) >> 4);
          const uint64_t off_b = (uint64_t)(((k >> 2) * (KV_TILE_BYTES / 2) + (k & 3) * 32) >> 4);
          ptx::mma_bf16_ss(d0 + COL_DP + pv.at * NKV, gd + off_a, vd0 + vtile + off_b, IDESC_S, k > 0 ? 1u : 0u);
        }
        ptx::mma_commit(bar(SD_FULL + pv.at));
      }
      __syncwarp();
    }
  } else {
    // =========================== issuer of dQ += dS K ===========================
    bool ok = true;
    int n_steps = 0x7fffffff;
    constexpr uint32_t IDESC_DQ = ptx::idesc_bf16_f32(128, HD, false, true);
    const uint64_t kmn0 = ptx::smem_desc_sw128(sbase + OFF_K, KV_TILE_BYTES / 2, 1024);   // K as MN-major B
    const uint32_t d0 = __shfl_sync(0xffffffffu, tmem, 0);
    RingPos<KST> pk;
    RingPos<VST> pv;
    for (int j = 0; j < n_steps && ok; ++j, pk.step(), pv.step()) {
      if (j == 1) {
        ok = wait_all(bar(META_READY), 0);
        if (!ok) break;
        n_steps = __shfl_sync(0xffffffffu, misc->n_steps, 0);
        if (j >= n_steps) break;
      }
      ok = wait_all(bar(DS_FULL + pv.at), pv.phase);
      if (!ok) break;
      ptx::tc_fence_after();
      const uint64_t kmn = kmn0 + (uint64_t)((pk.at * KV_TILE_BYTES) >> 4);
      // dS of keys 16k .. 16k+15: eight packed columns, keys 0-31 at columns 0-15 and keys 32-63 at columns 32-47 of the
      // step's S slot; the remainders, with two-term dS, 16 columns behind
      if (ptx::elect_one()) {
#pragma unroll
        for (int term = 0; term < (P2 ? 2 : 1); ++term)
#pragma unroll
          for (int k = 0; k < NKV / 16; ++k)
            ptx::mma_bf16_ts(d0 + COL_DQ, d0 + pv.at * NKV + (k >> 1) * 32 + term * 16 + (k & 1) * 8,
                             kmn + (uint64_t)((k * 16 * 128) >> 4), IDESC_DQ, (j > 0 || k > 0 || term > 0) ? 1u : 0u);
        ptx::mma_commit(bar(K_FREE + pk.at));
      }
      __syncwarp();
    }
  }
  } else {
    // =========================== dS / epilogue: thread = tile row, warpgroup wg takes the steps wg, wg + 3, ... ===========================
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(bwd_regs_row(WT, CPS)));
    const int wg = warp >> 2;
    const int m = (warp & 3) * 32 + lane;
    const int t = m / g_q, hh = m % g_q;
    const int i_row = i0 + t;
    const bool row_ok = i_row < dm.seq_q;
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const float c1 = dm.sm_scale * LOG2E;
    const float2 stat = row_ok ? *a.stats.at(b, r, i_row, hh) : make_float2(0.f, 0.f);
    const float lse2 = stat.x, delta = stat.y;
    float* drow = a.dbias + (long long)grp * dm.list_rows + list_row_offset(dm, min(i_row, dm.seq_q - 1));
    bool ok = true;
    int n_steps = 1;                       // step 0 always exists; the others are known with the walk
    if (wg > 0) {
      ok = wait_all(bar(META_READY), 0);
      n_steps = ok ? misc->n_steps : 0;
    }
    for (int j = wg; j < n_steps && ok; j += BWD_ROW_WG) {
      const int slot = j % VST, rec = j % KST;
      ok = wait_all(bar(REC_FULL + rec), (uint32_t)(j / KST) & 1u);    // the step's record is visible
      if (!ok) break;
      float off[CPS];                                      // -inf: the row did not route the chunk
      int pos[CPS], n_vis[CPS];                            // causal: column c of the slot visible iff c < n_vis
      bool any = false;
#pragma unroll
      for (int s = 0; s < CPS; ++s) {
        off[s] = row_ok ? misc->meta.bias[rec][s][t] * LOG2E - lse2 : -INFINITY;
        pos[s] = misc->meta.pos[rec][s][t];
        n_vis[s] = i_row - misc->meta.kvbase[rec][s] + 1;
        any = any || !(off[s] == -INFINITY);
      }
      any = __any_sync(0xffffffffu, any);                  // a warp none of whose rows routed a chunk of the step only writes zeros
      ok = wait_all(bar(SD_FULL + slot), (uint32_t)(j / VST) & 1u);
      if (!ok) break;
      ptx::tc_fence_after();
      float rowsum[CPS];
#pragma unroll
      for (int s = 0; s < CPS; ++s) rowsum[s] = 0.f;
#pragma unroll
      for (int half = 0; half < 2; ++half) {               // 32 columns at a time
        uint32_t hi[16], lo[16];
        if (any) {
          uint32_t sv[32], gv[32];
          DASH_TMEM_LD32(sv, lane_addr + slot * NKV + half * 32);
          DASH_TMEM_LD32(gv, lane_addr + COL_DP + slot * NKV + half * 32);
          DASH_TMEM_WAIT_LD32(sv);
          DASH_TMEM_WAIT_LD32(gv);
          float ds[32];
#pragma unroll
          for (int c = 0; c < 32; ++c) {
            const int s = (half * 32 + c) / W;
            const float p = half * 32 + c - s * W < n_vis[s] ? exp2f(fmaf(__uint_as_float(sv[c]), c1, off[s])) : 0.f;
            ds[c] = p * (__uint_as_float(gv[c]) - delta);
            rowsum[s] += ds[c];
          }
          // dS -> the first 16 columns of this half of the step's S slot (two bf16 per column), the remainders behind them
          pack_terms<P2>(ds, hi, lo);
        } else {
#pragma unroll
          for (int c = 0; c < 16; ++c) hi[c] = lo[c] = 0u;
        }
        ptx::tmem_st_n<16>(lane_addr + slot * NKV + half * 32, hi);
        if constexpr (P2) ptx::tmem_st_n<16>(lane_addr + slot * NKV + half * 32 + 16, lo);
      }
      ptx::tmem_wait_st();
      ptx::tc_fence_before();
      ptx::mbar_arrive(bar(DS_FULL + slot));
      // dbias of the (token, chunk): the row sums of the group's heads (adjacent lanes) added up
      if (any) {
#pragma unroll
        for (int s = 0; s < CPS; ++s) {
          for (int o = 1; o < g_q; o <<= 1) rowsum[s] += __shfl_xor_sync(0xffffffffu, rowsum[s], o);
          if (hh == 0 && pos[s] >= 0 && row_ok) atomicAdd(drow + pos[s], rowsum[s]);
        }
      }
      if (j == 0) {
        ok = wait_all(bar(META_READY), 0);
        n_steps = ok ? misc->n_steps : 0;
      }
    }
    // epilogue: dQ / sqrt(d) -> global; the warpgroups share the row's columns
    if (ok) {
      ok = wait_all(bar(META_READY), 0);
      n_steps = ok ? misc->n_steps : 0;
    }
    // (a warpgroup has seen the scores of step n-3 or a later one, or none where n < 3: the phase before this one is over)
    if (ok) ok = wait_all(bar(K_FREE + ((n_steps - 1) % KST)), (uint32_t)((n_steps - 1) / KST) & 1u);
    if (ok) {
      ptx::tc_fence_after();
      __nv_bfloat16* op = a.dQ + (long long)b * dm.qs[0] + (long long)i_row * dm.qs[1] + (long long)(r * g_q + hh) * dm.qs[2];
      const float sc = dm.sm_scale;
#pragma unroll 1
      for (int q = wg; q < HD / 32; q += BWD_ROW_WG) {
        uint32_t o[32];
        DASH_TMEM_LD32(o, lane_addr + COL_DQ + q * 32);
        ptx::tmem_wait_ld();
        if (row_ok) {
#pragma unroll
          for (int c = 0; c < 32; c += 8) {
            uint4 v;
            __nv_bfloat162 h0 = __floats2bfloat162_rn(__uint_as_float(o[c]) * sc, __uint_as_float(o[c + 1]) * sc);
            __nv_bfloat162 h1 = __floats2bfloat162_rn(__uint_as_float(o[c + 2]) * sc, __uint_as_float(o[c + 3]) * sc);
            __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(o[c + 4]) * sc, __uint_as_float(o[c + 5]) * sc);
            __nv_bfloat162 h3 = __floats2bfloat162_rn(__uint_as_float(o[c + 6]) * sc, __uint_as_float(o[c + 7]) * sc);
            v.x = *reinterpret_cast<uint32_t*>(&h0); v.y = *reinterpret_cast<uint32_t*>(&h1);
            v.z = *reinterpret_cast<uint32_t*>(&h2); v.w = *reinterpret_cast<uint32_t*>(&h3);
            *reinterpret_cast<uint4*>(op + q * 32 + c) = v;
          }
        }
      }
    }
    ptx::tc_fence_before();
  }

  __syncthreads();
  if (warp == BWD_W_SD) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, TMEM_COLS);
  }
  if (misc->abort_flag) {
    // nothing of what the gradient buffers held as scratch may pass for a gradient
    const __nv_bfloat162 nan2 = __floats2bfloat162_rn(gave_up(), gave_up());
    for (int k = tid; k < 128 * HD / 2; k += THREADS) {
      const int m = k / (HD / 2), i = i0 + m / g_q;
      if (i < dm.seq_q)
        *reinterpret_cast<__nv_bfloat162*>(a.dQ + (long long)b * dm.qs[0] + (long long)i * dm.qs[1] + (long long)(r * g_q + m % g_q) * dm.qs[2] + 2 * (k % (HD / 2))) = nan2;
    }
    const long long at = (long long)grp * dm.list_rows, hi = i0 + TQ < dm.seq_q ? list_row_offset(dm, i0 + TQ) : dm.list_rows;
    for (long long k = list_row_offset(dm, i0) + tid; k < hi; k += THREADS) a.dbias[at + k] = gave_up();
  }
  if (tid == 0 && misc->abort_flag) report_error(a.sb, DASH_ERR_TIMEOUT, 111);
}

}  // namespace dq

// ===================================================================================================================
// dK and dV: key-slice stationary
// ===================================================================================================================
namespace dkv {

// Two warpgroups form P and dS, each for half of the slice's keys on every step (no row maximum is needed, so the halves
// are independent and a step's P / dS stretch takes half as long); one issuing thread per product: 32 MMAs per step
// are too many for one.  W_SCAN reads the slice's column of the mask and collects the tokens that attend the slice; the
// loader warps copy their rows, 16 bytes per lane; W_META looks up their biases and statistics.  W_SD issues S, W_DP dP, W_ACC
// dV^T, W_DK dK^T.
// 8192 tokens, 32/8 heads, chunks of 64, 29 % of the chunks routed: whole query tiles of 32 tokens, of which one in two has a
// token for the slice, 87.8 K steps and 1.05 ms; gathered 37.7 K steps and 0.57 ms.  A TMA box per token and half row instead of the
// copies: 27 clocks of the TMA unit each, 128 of them a step, 0.85 ms.  The seven roles share an instruction cache: with the
// scanner's and loaders' loops unrolled eight to sixteen times every role slows down, 0.77-1.15 ms.
constexpr int W_SD = 8, W_ACC = 9, W_DP = 10, W_DK = 11, W_META = 12, W_SCAN = 13;
// Loaders: four in a warpgroup of their own; two-term kernels, whose P / dS threads keep 64 sums, make do with the two warps left.
__host__ __device__ constexpr int n_load(bool p2) { return p2 ? 2 : 4; }
__host__ __device__ constexpr int w_load(bool p2) { return p2 ? 14 : 16; }
__host__ __device__ constexpr int threads(bool p2) { return p2 ? 512 : 640; }
// registers per thread after the re-division (at launch: 128 with two terms, 96 with one)
__host__ __device__ constexpr int regs_service(bool p2, int tpl) { return p2 ? (tpl > 2 ? 96 : 80) : 64; }
__host__ __device__ constexpr int regs_rows(bool p2, int tpl) { return p2 ? 256 - regs_service(p2, tpl) : 144; }
static_assert(2 * regs_rows(false, 2) + 3 * regs_service(false, 2) <= 5 * 96, "the block's own pool is all that it can draw from");
constexpr uint32_t TMEM_COLS = 512;     // S0 S1 [0,128) dP0 dP1 [128,256) dV^T [256,320) dK^T [320,384)
constexpr uint32_t COL_DP = 128, COL_DV = 256, COL_DK = 320;
constexpr uint32_t PS_BYTES = 128 * NKV * 2;       // 16 KiB: one term of P (or dS) of a step, 128 rows of 128 bytes
constexpr int MAX_STAGES = 4, MAX_SLOTS = 16, AHEAD = 16;
// Two-term kernels take their sums out of tensor memory every FLUSH steps and add them up in registers: the tensor cores cut the
// low bits of an accumulator off at every product, so that a sum left there loses about half a unit per product, the longer
// the walk the more.  dK against float64, 16 heads per KV head, d 64 (relative 2-norm): 1500 tokens 1.3e-5 -> 2.5e-6, 6000
// tokens 2.8e-4 -> 2.3e-6, which is the two terms' own 2^-18; 2 x 1500 tokens, 8/2 heads: 152.9 -> 154.7 us the whole backward.
constexpr int FLUSH = 2;
// SD_FULL: both score products of the step (two arrivals).  PDS_FULL: P and dS in shared memory (SEQ: P alone).
// ACC_DONE: both accumulating products done (SEQ: dK, which follows dV), the step's stage and the P / dS buffers are free.
// TOK_FULL / TOK_FREE: a step's tokens are listed / have been read by W_PROD and W_META.
enum Bar { KV_FULL = 0, SD_FULL = 1, PDS_FULL = 3, DV_DONE = 5, DS_FULL = 7, QD_FULL = 9, ACC_DONE = 9 + MAX_STAGES,
           TOK_FULL = 9 + 2 * MAX_STAGES, TOK_FREE = TOK_FULL + MAX_SLOTS, N_BARS = TOK_FREE + MAX_SLOTS };

// A stage holds a Q and a dO tile.  head_dim 128: two stages, Q then dO.  head_dim 64: four stages, dO then Q, so that the
// two tiles read as MN-major A stack to the M = 128 rows that an accumulating product needs: lanes 0-63 of dO^T P are
// dV^T, lanes 64-127 of Q^T dS are dK^T (the other halves are not used).
// Two-term P and dS (P2) take four buffers; at head_dim 128 only two fit, so there dS follows P through the same pair
// once the dV product has read it (SEQ).
template <int HD, int CPS, int MTQ, bool P2>
struct Layout {
  static constexpr int NST = HD == 128 ? 2 : 4;
  static constexpr bool SEQ = P2 && HD == 128;
  static constexpr int LOG_RING = MTQ > 64 ? 8 : 7, RING = 1 << LOG_RING;      // tokens that W_SCAN is ahead: 2 steps of MTQ tokens .. 16 of 8
  struct Misc {
    unsigned long long bar[N_BARS];
    uint32_t tmem_base;
    int abort_flag;
    int total;                            // number of steps, written with the end marker
    int live[NST];                        // the stage holds a step, 1 with gathered rows, 0 without; -1: no more steps
    int irow[NST][MTQ];                   // token of each of the step's rows
    float bias[NST][CPS][MTQ];            // per token of the step: the chunk's bias (-inf: the token does not attend it)
    // what W_SCAN hands on: tokens (bit 31: a repetition that fills up the last step) and their mask words over the slice's
    // chunks, step after step; last[slot]: no such step
    int tok[RING], last[MAX_SLOTS];
    uint32_t word[RING];
    uint32_t whole[MAX_SLOTS];            // the step's runs that are consecutive tokens (a bit each)
    uint32_t ahead[AHEAD][32];            // mask words that W_SCAN has asked for
    alignas(16) float2 stats[NST][128];   // log-sum-exp and delta of the tile's rows
  };
  static constexpr uint32_t Q_BYTES = 128 * HD * 2, KV_TILE_BYTES = NKV * HD * 2, STAGE = 2 * Q_BYTES;
  static constexpr uint32_t AT_Q = HD == 128 ? 0 : Q_BYTES, AT_G = HD == 128 ? Q_BYTES : 0;     // inside a stage
  static constexpr uint32_t OFF_K = 0, OFF_V = OFF_K + KV_TILE_BYTES, OFF_ST = OFF_V + KV_TILE_BYTES,
                            OFF_P = OFF_ST + NST * STAGE,                        // terms hi (, lo) of P, then of dS
                            OFF_DS = SEQ ? OFF_P : OFF_P + (P2 ? 2 : 1) * PS_BYTES,
                            OFF_MISC = OFF_P + (P2 && !SEQ ? 4 : 2) * PS_BYTES, SMEM = OFF_MISC + sizeof(Misc);
  static_assert(SMEM <= 232448, "one block per SM");
};

// TPL: tokens per lane of the service warps, a step's tokens being at most 32 * TPL.
template <int HD, int CPS, int TPL, bool P2>
__global__ void __launch_bounds__(threads(P2), 1)
attend_bwd_dkv_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmDO,
                      const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, BwdArgs a) {
  constexpr int NLOAD = n_load(P2), W_LOAD = w_load(P2), THREADS = threads(P2);
  constexpr int MTQ = 32 * TPL;
  using LY = Layout<HD, CPS, MTQ, P2>;
  using Misc = typename LY::Misc;
  constexpr int NST = LY::NST;
  constexpr bool SEQ = LY::SEQ;
  constexpr uint32_t Q_BYTES = LY::Q_BYTES, KV_TILE_BYTES = LY::KV_TILE_BYTES, OFF_K = LY::OFF_K, OFF_V = LY::OFF_V;
  extern __shared__ __align__(1024) uint8_t smem[];
  Misc* misc = reinterpret_cast<Misc*>(smem + LY::OFF_MISC);
  const Dims& dm = a.dm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t sbase = ptx::smem_u32(smem);
  auto bar = [&](int i) { return ptx::smem_u32(&misc->bar[i]); };
  volatile int* abort_flag = &misc->abort_flag;
  const long long wait_limit = a.wait_limit;
  auto wait_on = [&](uint32_t barrier, uint32_t parity) { return ptx::mbar_wait(barrier, parity, abort_flag, wait_limit); };
  auto wait_all = [&](uint32_t barrier, uint32_t parity) { return ptx::mbar_wait_warp(barrier, parity, abort_flag, wait_limit); };

  const int groups = dm.batch * dm.h_kv;
  const int slice = (int)(blockIdx.x / groups);                  // early slices first: every later token may attend them
  const int grp = (int)(blockIdx.x % groups);
  const int b = grp / dm.h_kv, r = grp % dm.h_kv;
  const int TQ = a.TQ, g_q = dm.g_q;
  const int k0 = slice * NKV;                                    // first key of the slice
  const int c = k0 >> dm.log_b;                                       // its first chunk (CPS of them)
  const int log_t = 31 - __clz(TQ), log_slots = LY::LOG_RING - log_t, n_slots = 1 << log_slots;      // a step has TQ tokens; steps in W_SCAN's ring (2 .. 16)
  const int log_run = min(log_t, 5), log_rps = log_t - log_run;      // tokens of a run, runs of a step (1, 2 or 4)

  if (tid == 0) {
    misc->abort_flag = ((sbase & 1023u) != 0u) ? 1 : 0;
    if (misc->abort_flag) report_error(a.sb, DASH_ERR_CUDA, 120);
    ptx::mbar_init(bar(KV_FULL), 1);
    for (int s = 0; s < NST; ++s) {
      // one arrival of the first loader, one of W_META, and one per lane of the loaders for the copies in flight
      ptx::mbar_init(bar(QD_FULL + s), 2 + 32 * NLOAD);
      ptx::mbar_init(bar(ACC_DONE + s), SEQ ? 1 : 2);
    }
    for (int s = 0; s < n_slots; ++s) {
      misc->last[s] = 0;
      ptx::mbar_init(bar(TOK_FULL + s), 1);
      ptx::mbar_init(bar(TOK_FREE + s), NLOAD + 1);
    }
    for (int s = 0; s < 2; ++s) {
      ptx::mbar_init(bar(SD_FULL + s), 2);
      ptx::mbar_init(bar(PDS_FULL + s), 256);
      ptx::mbar_init(bar(DV_DONE + s), 1);
      ptx::mbar_init(bar(DS_FULL + s), 256);
    }
    ptx::fence_barrier_init();
  }
  if (warp == W_SD) {
    ptx::tmem_alloc(ptx::smem_u32(&misc->tmem_base), TMEM_COLS);
    ptx::tmem_relinquish();
    ptx::tc_fence_before();
  }
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = misc->tmem_base;
  chain_wait();
  chain_release();
  if (a.sb && *reinterpret_cast<volatile int*>(&a.sb->status) != 0) *abort_flag = 1;
  __syncthreads();

  if (warp >= 8) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(regs_service(P2, TPL)));
  const int wc = c >> 5, bit = c & 31;             // (the slice's chunks share a mask word)
  const long long row0 = (long long)grp * dm.seq_q;
  if (warp == W_SCAN) {
    // =========================== scanner ===========================
    // The tokens from k0 on, 32 at a time, the mask words of the next groups on their way; those that attend the
    // slice (its own chunks' tokens, and later ones that routed one of them) are appended to the ring.  A run of neighbours most of which
    // attend it goes in as it is, in front of the run that is being gathered: the loader fetches it with one copy per tensor.
    // With several blocks per slice, block s takes every n_split-th group.  (A short loop on purpose: one warp that runs
    // through unrolled code waits for its instructions, and pushes the other roles' out of the cache.)
    const int stride = 32 * a.n_split, R = 1 << log_run;
    bool ok = true;
    int n = 0, free_slots = n_slots, done = 0;      // tokens so far; steps that may be written; steps handed on
    uint32_t marks = 0u;                            // the open step's runs that are neighbours
    auto reserve = [&](int steps) {
      for (; free_slots < steps && ok; ++free_slots)
        ok = wait_all(bar(TOK_FREE + (free_slots & (n_slots - 1))), (uint32_t)((free_slots >> log_slots) - 1) & 1u);
    };
    auto hand_on = [&](int steps) {
      __syncwarp();
      if (lane == 0)
        for (int k = done; k < steps; ++k) {
          misc->whole[k & (n_slots - 1)] = k == done ? marks : 0u;
          ptx::mbar_arrive(bar(TOK_FULL + (k & (n_slots - 1))));
        }
      done = steps;
      marks = 0u;
    };
    const int i_first = k0 + 32 * (int)blockIdx.y + lane;
    const uint32_t* src = a.mask + (row0 + i_first) * dm.W + wc;
    const long long src_step = (long long)stride * dm.W;
    const uint32_t ahead = ptx::smem_u32(&misc->ahead[0][lane]);
    int i_next = i_first;                           // token whose word is asked for next
    uint32_t g = 0;                                 // groups looked at
    auto ask = [&](uint32_t group) {
      if (i_next < dm.seq_q) copy_async4(ahead + (group & (AHEAD - 1)) * 128, src);
      asm volatile("cp.async.commit_group;" ::: "memory");
      src += src_step;
      i_next += stride;
    };
#pragma unroll 1
    for (uint32_t k = 0; k < AHEAD - 1; ++k) ask(k);
#pragma unroll 1
    for (int i = i_first; i - lane < dm.seq_q && ok; i += stride, ++g) {
      ask(g + AHEAD - 1);
      asm volatile("cp.async.wait_group %0;" ::"n"(AHEAD - 1) : "memory");
      const uint32_t word = misc->ahead[g & (AHEAD - 1)][lane];      // (only this lane wrote it)
      const int own = i >> dm.log_b;
      bool on = false;
#pragma unroll
      for (int s = 0; s < CPS; ++s) on = on || c + s == own || (c + s < own && ((word >> (bit + s)) & 1u));
      const uint32_t hit = __ballot_sync(0xffffffffu, on && i < dm.seq_q);
      if (hit == 0u) continue;
      const int n_hit = __popc(hit);
      // (a gathered row costs about 1.25 rows of a run that is fetched as it is)
      if (5 * n_hit < 4 * R || i - lane + 32 > dm.seq_q) {
        const int e = (n + __popc(hit & ((1u << lane) - 1u))) & (LY::RING - 1);
        n += n_hit;
        reserve(((n - 1) >> log_t) + 1);
        if ((hit >> lane) & 1u) {
          misc->tok[e] = i;
          misc->word[e] = word;
        }
        if ((n >> log_t) > done) hand_on(n >> log_t);
        continue;
      }
#pragma unroll 1
      for (int at = 0; at < 32 && ok; at += R) {
        const uint32_t bits = (hit >> at) & (0xffffffffu >> (32 - R));
        const bool here = (unsigned)(lane - at) < (unsigned)R;
        const int first = n & ~(R - 1), open = n - first;
        const bool whole = 5 * __popc(bits) >= 4 * R;
        int e = n + __popc(bits & ((1u << ((lane - at) & 31)) - 1u)), tok = 0;
        uint32_t w = 0u;
        if (whole) {                                // the run being gathered moves on by one, and this one takes its place
          if (lane < open) {
            tok = misc->tok[(first + lane) & (LY::RING - 1)];
            w = misc->word[(first + lane) & (LY::RING - 1)];
          }
          e = first + lane - at;
          marks |= 1u << ((first >> log_run) & ((1 << log_rps) - 1));
        }
        n += whole ? R : __popc(bits);
        reserve(((n - 1) >> log_t) + 1);
        __syncwarp();
        if (whole && lane < open) {
          misc->tok[(first + R + lane) & (LY::RING - 1)] = tok;
          misc->word[(first + R + lane) & (LY::RING - 1)] = w;
        }
        if (here && (whole || ((hit >> lane) & 1u))) {
          misc->tok[e & (LY::RING - 1)] = i;
          misc->word[e & (LY::RING - 1)] = word;
        }
        if ((n >> log_t) > done) hand_on(n >> log_t);
      }
    }
    const int steps = (n + TQ - 1) >> log_t;
    if (ok && steps > done) {                       // fill up the last step with copies of a token whose weights will be zero
      __syncwarp();
      const int copy = misc->tok[(done << log_t) & (LY::RING - 1)] | (int)0x80000000;
#pragma unroll 1
      for (int e = n + lane; e < steps << log_t; e += 32) {
        misc->tok[e & (LY::RING - 1)] = copy;
        misc->word[e & (LY::RING - 1)] = 0u;
      }
      hand_on(steps);
    }
    reserve(steps + 1);
    if (ok && lane == 0) {
      misc->last[steps & (n_slots - 1)] = 1;
      ptx::mbar_arrive(bar(TOK_FULL + (steps & (n_slots - 1))));
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else if (warp >= W_LOAD && warp < W_LOAD + NLOAD) {
    // =========================== loaders ===========================
    // The first one fetches K / V and the Q / dO rows of runs of neighbours, all of them the rows of gathered tokens: a lane copies one
    // 16-byte piece of a row, to where the 128-byte swizzle has it.  A step's stage is free once both accumulating products of the
    // step NST before have completed.  (cp.async writes through the generic proxy: the issuers fence before their products read
    // the stage.)
    constexpr int PIECES = HD / 8, RP = 32 / PIECES;      // pieces of a row, rows of a warp's copy
    constexpr int NR = 16 / (RP * NLOAD);                 // of sixteen rows at a time, a loader copies NR x RP
    const int w = warp - W_LOAD, p = lane % PIECES;
    if (w == 0 && lane == 0) {
      ptx::prefetch_tensormap(&tmQ);
      ptx::prefetch_tensormap(&tmDO);
      ptx::prefetch_tensormap(&tmK);
      ptx::prefetch_tensormap(&tmV);
      ptx::mbar_arrive_expect_tx(bar(KV_FULL), 2 * KV_TILE_BYTES);
      ptx::tma_load_4d(sbase + OFF_K, &tmK, bar(KV_FULL), 0, r, k0, b);
      if constexpr (HD == 128) ptx::tma_load_4d(sbase + OFF_K + KV_TILE_BYTES / 2, &tmK, bar(KV_FULL), 64, r, k0, b);
      ptx::tma_load_4d(sbase + OFF_V, &tmV, bar(KV_FULL), 0, r, k0, b);
      if constexpr (HD == 128) ptx::tma_load_4d(sbase + OFF_V + KV_TILE_BYTES / 2, &tmV, bar(KV_FULL), 64, r, k0, b);
    }
    // (sixteen rows on, a row has the same head of the group and the same place in the swizzle)
    const char *q0[NR], *g0[NR];
    uint32_t dst0[NR], tok0[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      const int m = (w + k * NLOAD) * RP + lane / PIECES, head = r * g_q + (m & (g_q - 1));
      q0[k] = reinterpret_cast<const char*>(a.Q + (long long)b * dm.qs[0] + head * dm.qs[2] + p * 8);
      g0[k] = reinterpret_cast<const char*>(a.dO + (long long)b * dm.os[0] + head * dm.os[2] + p * 8);
      dst0[k] = sbase + LY::OFF_ST + (p >> 3) * (Q_BYTES / 2) + m * 128 + (((p ^ m) & 7) << 4);
      tok0[k] = m / g_q;
    }
    const long long q_tok = dm.qs[1] * 2, g_tok = dm.os[1] * 2;
    bool ok = true;
    int n_done = 0;                                       // steps whose copies are under way
    for (int j = 0;; ++j) {
      const int st = j % NST, sl = j & (n_slots - 1);
      ok = wait_all(bar(TOK_FULL + sl), (uint32_t)(j >> log_slots) & 1u);
      if (!ok) break;
      const bool end = *reinterpret_cast<volatile int*>(&misc->last[sl]) != 0;
      const uint32_t whole = end ? 0u : *reinterpret_cast<volatile uint32_t*>(&misc->whole[sl]);
      const uint32_t tx = 2 * (Q_BYTES >> log_rps) * __popc(whole);
      int first = misc->tok[sl << log_t];                       // (of the first run)
      if (j >= NST) ok = wait_all(bar(ACC_DONE + st), (uint32_t)(j / NST - 1) & 1u);
      if (!ok) break;
      if (w == 0 && lane == 0) {
        misc->live[st] = end ? -1 : whole != (2u << ((1 << log_rps) - 1)) - 1u;
        if (end) misc->total = j;
        if (whole == 0u) ptx::mbar_arrive(bar(QD_FULL + st));
        else ptx::mbar_arrive_expect_tx(bar(QD_FULL + st), tx);
        for (int run = 0; whole >> run; ++run) {
          if (run > 0) first = misc->tok[(sl << log_t) + (run << log_run)];
          if (!((whole >> run) & 1u)) continue;
          const uint32_t dst = sbase + LY::OFF_ST + st * LY::STAGE + run * (128 >> log_rps) * 128;
#pragma unroll
          for (int h = 0; h < HD / 64; ++h) {
            ptx::tma_load_4d(dst + LY::AT_Q + h * (Q_BYTES / 2), &tmQ, bar(QD_FULL + st), 64 * h, r * g_q, first, b);
            ptx::tma_load_4d(dst + LY::AT_G + h * (Q_BYTES / 2), &tmDO, bar(QD_FULL + st), 64 * h, r * g_q, first, b);
          }
        }
      }
      if (!end) {
        const int per_run = 8 >> log_rps;                  // times sixteen rows
#pragma unroll 1
        for (int run = 0; run < 1 << log_rps; ++run) {
          if ((whole >> run) & 1u) continue;
          uint32_t at = st * LY::STAGE + run * per_run * 16 * 128;
          const int* t = misc->tok + (sl << log_t) + (run << log_run);
#pragma unroll 1
          for (int it = 0; it < per_run; ++it, at += 16 * 128, t += 16 / g_q) {
            uint32_t i[NR];
#pragma unroll
            for (int k = 0; k < NR; ++k) i[k] = (uint32_t)t[tok0[k]] & 0x7fffffffu;
#pragma unroll
            for (int k = 0; k < NR; ++k) {
              copy_async16(dst0[k] + at + LY::AT_Q, q0[k] + (unsigned long long)i[k] * q_tok);
              copy_async16(dst0[k] + at + LY::AT_G, g0[k] + (unsigned long long)i[k] * g_tok);
            }
          }
        }
      }
      arrive_after_copies(bar(QD_FULL + st));
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(bar(TOK_FREE + sl));
      if (end) break;
      n_done = j + 1;
    }
    // a wait that ran out: the copies already issued land before the block retires
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (!ok && w == 0 && lane == 0) {
      for (int k = 0; k < 200000 && !ptx::mbar_try_wait(bar(KV_FULL), 0); ++k) {}
      for (int j = max(n_done - NST, 0); j < n_done; ++j)
        for (int k = 0; k < 200000 && !ptx::mbar_try_wait(bar(QD_FULL + j % NST), (uint32_t)(j / NST) & 1u); ++k) {}
    }
  } else if (warp == W_META) {
    // =========================== biases and statistics of every step ===========================
    // A bias is behind two loads in a row: the count of the row's routed chunks before the slice's mask word, and the list entry.  Each
    // has a step's time: while step j is stored, the counts of step j + 1 are under way (if its tokens are listed by then), and
    // its biases and statistics are asked for once step j has been handed on.  (One step after the other this warp was the pace of the
    // kernel, 3300 clk a step at 8192 tokens, 32/8 heads, chunks of 64, all of them routed, 5700-6300 with 128 tokens a step; loads,
    // because an asynchronous copy to 32 places holds the warp up for some 200 clk.)
    const long long list0 = (long long)grp * dm.list_rows;
    int tok[TPL], before[TPL];           // tokens of the next step, routed chunks before the slice's mask word
    uint32_t word[TPL];
    long long at[TPL];                   // start of the token's list
    int i_now[TPL];                      // tokens, biases and statistics of this step
    float bias[CPS][TPL];
    float2 stat[4];
    int n_tok = 0;                       // steps whose tokens have been read
    bool end = false;                    // the last of them is the end marker
    // this lane's rows: lane + 32 k
    const char* stat0 = reinterpret_cast<const char*>(a.stats.at(b, r, 0, 0));
    uint32_t stat_at[4], stat_tok[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      stat_tok[k] = (lane + 32 * k) / g_q;
      stat_at[k] = (uint32_t)(((lane + 32 * k) & (g_q - 1)) * a.stats.sh);
    }
    auto read_tokens = [&]() {
      const int sl = n_tok++ & (n_slots - 1);
      end = *reinterpret_cast<volatile int*>(&misc->last[sl]) != 0;
      if (end) return;
#pragma unroll
      for (int q = 0; q < TPL; ++q) {
        if (32 * q >= TQ) break;
        const bool in = lane + 32 * q < TQ;
        const int e = (sl << log_t) + lane + 32 * q;
        tok[q] = in ? misc->tok[e] : (int)0x80000000;
        word[q] = in ? misc->word[e] : 0u;
        at[q] = list0 + list_row_offset(dm, tok[q] & 0x7fffffff);
        before[q] = wc > 0 && tok[q] >= 0 && (tok[q] >> dm.log_b) > c ? a.marks[at[q] + wc - 1] : 0;
      }
    };
    bool ok = true;
    for (int j = 0; ok; ++j) {
      const int st = j % NST, sl = j & (n_slots - 1);
      if (n_tok == j) {
        ok = wait_all(bar(TOK_FULL + sl), (uint32_t)(j >> log_slots) & 1u);
        if (!ok) break;
        read_tokens();
      }
      const bool last = end;
      if (!last) {
#pragma unroll
        for (int q = 0; q < TPL; ++q) {
          if (32 * q >= TQ) break;
          const int own = (tok[q] & 0x7fffffff) >> dm.log_b;
          const float* entry = a.blk_bias + at[q] + before[q];
          i_now[q] = tok[q] & 0x7fffffff;
#pragma unroll
          for (int s = 0; s < CPS; ++s) {
            bias[s][q] = tok[q] >= 0 && c + s == own ? 0.f : -INFINITY;
            if (tok[q] >= 0 && c + s < own && ((word[q] >> (bit + s)) & 1u)) bias[s][q] = __ldg(entry + __popc(word[q] & ((1u << (bit + s)) - 1u)));
          }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
          stat[k] = *reinterpret_cast<const float2*>(stat0 + (long long)(misc->tok[(sl << log_t) + stat_tok[k]] & 0x7fffffff) * a.stats.si + stat_at[k]);
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(bar(TOK_FREE + sl));
        if (__all_sync(0xffffffffu, ptx::mbar_test_wait(bar(TOK_FULL + ((j + 1) & (n_slots - 1))), (uint32_t)((j + 1) >> log_slots) & 1u))) read_tokens();
      }
      if (j >= NST) ok = wait_all(bar(ACC_DONE + st), (uint32_t)(j / NST - 1) & 1u);
      if (!ok) break;
      if (!last) {
#pragma unroll
        for (int q = 0; q < TPL; ++q) {
          const int t = lane + 32 * q;
          if (t < TQ) {
            misc->irow[st][t] = i_now[q];
#pragma unroll
            for (int s = 0; s < CPS; ++s) misc->bias[st][s][t] = bias[s][q];
          }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) misc->stats[st][lane + 32 * k] = stat[k];
      }
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(bar(QD_FULL + st));
      if (last) break;
    }
  } else if (warp == W_SD || warp == W_DP) {
    // =========================== issuers of the score products: S = Q K^T (W_SD), dP = dO V^T (W_DP) ===========================
    if (lane == 0) {
      const bool is_s = warp == W_SD;
      bool ok = wait_on(bar(KV_FULL), 0);
      constexpr uint32_t IDESC_S = ptx::idesc_bf16_f32(128, NKV, false, false);
      const uint64_t bd0 = ptx::smem_desc_sw128(sbase + (is_s ? OFF_K : OFF_V), 16, 1024);
      const uint32_t col0 = is_s ? 0u : COL_DP;
      for (int j = 0; ok; ++j) {
        const int buf = j & 1, st = j % NST;
        ok = wait_on(bar(QD_FULL + st), (uint32_t)(j / NST) & 1u);
        const int live = ok ? *reinterpret_cast<volatile int*>(&misc->live[st]) : -1;
        if (live < 0) break;
        if (live > 0) ptx::fence_proxy_async_smem();
        // the P / dS warps have read S / dP of step j-2
        if (j >= 2) ok = wait_on(bar(PDS_FULL + buf), (uint32_t)((j >> 1) - 1) & 1u);
        if (!ok) break;
        ptx::tc_fence_after();
        const uint64_t ad0 = ptx::smem_desc_sw128(sbase + LY::OFF_ST + st * LY::STAGE + (is_s ? LY::AT_Q : LY::AT_G), 16, 1024);
#pragma unroll
        for (int k = 0; k < HD / 16; ++k) {
          const uint64_t off_a = (uint64_t)(((k >> 2) * (Q_BYTES / 2) + (k & 3) * 32) >> 4);
          const uint64_t off_b = (uint64_t)(((k >> 2) * (KV_TILE_BYTES / 2) + (k & 3) * 32) >> 4);
          ptx::mma_bf16_ss(tmem + col0 + buf * NKV, ad0 + off_a, bd0 + off_b, IDESC_S, k > 0 ? 1u : 0u);
        }
        ptx::mma_commit(bar(SD_FULL + buf));
      }
    }
    __syncwarp();
  } else if (warp == W_ACC || warp == W_DK) {
    // =========================== issuers of the accumulating products: dV^T += dO^T P (W_ACC), dK^T += Q^T dS (W_DK) ===========================
    if (lane == 0) {
      const bool is_v = warp == W_ACC;
      constexpr uint32_t IDESC_ACC = ptx::idesc_bf16_f32(128, NKV, true, true);     // A = (Q | dO)^T, B = (dS | P): both MN-major
      const uint64_t bd0 = ptx::smem_desc_sw128(sbase + (is_v ? LY::OFF_P : LY::OFF_DS), PS_BYTES, 1024);
      const uint32_t d_tmem = tmem + (is_v ? COL_DV : COL_DK);
      bool ok = true;
      for (int j = 0; ok; ++j) {
        const int buf = j & 1, st = j % NST;
        ok = wait_on(bar(QD_FULL + st), (uint32_t)(j / NST) & 1u);
        const int live = ok ? *reinterpret_cast<volatile int*>(&misc->live[st]) : -1;
        if (live < 0) break;
        if (live > 0) ptx::fence_proxy_async_smem();
        ok = wait_on(bar((SEQ && !is_v ? DS_FULL : PDS_FULL) + buf), (uint32_t)(j >> 1) & 1u);
        if (!ok) break;
        ptx::tc_fence_after();
        // tile [row][d] read as MN-major A: M = d (two blocks of 64), K = rows (16 rows = 2048 B); at head_dim 64 the two
        // blocks are the dO and the Q tile
        const uint64_t ad0 = ptx::smem_desc_sw128(sbase + LY::OFF_ST + st * LY::STAGE + (HD == 64 ? 0 : is_v ? LY::AT_G : LY::AT_Q),
                                                  HD == 64 ? Q_BYTES : Q_BYTES / 2, 1024);
#pragma unroll
        for (int term = 0; term < (P2 ? 2 : 1); ++term)
#pragma unroll
          for (int k = 0; k < 128 / 16; ++k) {
            const uint64_t adv = (uint64_t)((k * 16 * 128) >> 4);
            ptx::mma_bf16_ss(d_tmem, ad0 + adv, bd0 + adv + (uint64_t)((term * PS_BYTES) >> 4), IDESC_ACC,
                             ((P2 ? j % FLUSH : j) > 0 || k > 0 || term > 0) ? 1u : 0u);
          }
        ptx::mma_commit(SEQ && is_v ? bar(DV_DONE + buf) : bar(ACC_DONE + st));
      }
    }
    __syncwarp();
  }
  } else {
    // =========================== P, dS: thread = tile row, warpgroup = half of the keys; epilogue: thread = d ===========================
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(regs_rows(P2, TPL)));
    constexpr int SPH = CPS == 4 ? 2 : 1;                  // chunks in a half of the slice
    const int wg = warp >> 2;
    const int m = (warp & 3) * 32 + lane;
    const int t = m / g_q;
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const float c1 = dm.sm_scale * LOG2E;
    const bool mine = HD == 128 || (wg == 0 ? m < 64 : m >= 64);      // this thread's lane holds sums (whole warps)
    const uint32_t sum_addr = lane_addr + (wg == 0 ? COL_DV : COL_DK);
    [[maybe_unused]] float sums[P2 ? NKV : 1];                        // dV or dK of row d = lane, one per key
    if constexpr (P2) {
#pragma unroll
      for (int cc = 0; cc < NKV; ++cc) sums[cc] = 0.f;
    }
    [[maybe_unused]] auto take_sums = [&]() {
      if constexpr (P2) {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          uint32_t v[32];
          DASH_TMEM_LD32(v, sum_addr + half * 32);
          ptx::tmem_wait_ld();
#pragma unroll
          for (int cc = 0; cc < 32; ++cc) sums[half * 32 + cc] += __uint_as_float(v[cc]);
        }
      }
    };
    bool ok = true;
    // row m of a [128 rows][64 keys] term: 128 bytes, 16-byte pieces swizzled with the row (128-byte swizzle); this
    // warpgroup's keys are pieces 4 wg .. 4 wg + 3
    auto store_row = [&](uint32_t off, const uint32_t (&v)[16]) {
      uint8_t* row = smem + off + m * 128;
#pragma unroll
      for (int ch = 0; ch < 4; ++ch)
        *reinterpret_cast<uint4*>(row + (((wg * 4 + ch) ^ (m & 7)) << 4)) = make_uint4(v[ch * 4], v[ch * 4 + 1], v[ch * 4 + 2], v[ch * 4 + 3]);
    };
    for (int j = 0; ok; ++j) {
      const int buf = j & 1, st = j % NST;
      const uint32_t ph = (uint32_t)(j >> 1) & 1u;
      ok = wait_all(bar(QD_FULL + st), (uint32_t)(j / NST) & 1u);
      if (!ok) break;
      if (*reinterpret_cast<volatile int*>(&misc->live[st]) < 0) break;
      const int i_row = misc->irow[st][t];
      const float2 stat = misc->stats[st][m];
      const float lse2 = stat.x, delta = stat.y;
      float off[SPH];
#pragma unroll
      for (int s = 0; s < SPH; ++s) off[s] = misc->bias[st][CPS == 1 ? 0 : wg * SPH + s][t] * LOG2E - lse2;
      const int n_vis = i_row - k0 + 1 - wg * 32;            // visible columns of this warpgroup's half
      ok = wait_all(bar(SD_FULL + buf), ph);
      if (!ok) break;
      ptx::tc_fence_after();
      uint32_t p_hi[16], p_lo[16], d_hi[16], d_lo[16];       // the row's 32 P and 32 dS values of this half as bf16 pairs
      {
        uint32_t sv[32], gv[32];
        DASH_TMEM_LD32(sv, lane_addr + buf * NKV + wg * 32);
        DASH_TMEM_LD32(gv, lane_addr + COL_DP + buf * NKV + wg * 32);
        ptx::tmem_wait_ld();
        float p[32], ds[32];
#pragma unroll
        for (int cc = 0; cc < 32; ++cc) {
          p[cc] = cc < n_vis ? exp2f(fmaf(__uint_as_float(sv[cc]), c1, off[cc / (32 / SPH)])) : 0.f;
          ds[cc] = p[cc] * (__uint_as_float(gv[cc]) - delta);
        }
        pack_terms<P2>(p, p_hi, p_lo);
        pack_terms<P2>(ds, d_hi, d_lo);
      }
      // the accumulating products of the step before have read P / dS
      if (j >= 1) ok = wait_all(bar(ACC_DONE + (j - 1) % NST), (uint32_t)((j - 1) / NST) & 1u);
      if (!ok) break;
      store_row(LY::OFF_P, p_hi);
      if constexpr (P2) store_row(LY::OFF_P + PS_BYTES, p_lo);
      if constexpr (!SEQ) {
        store_row(LY::OFF_DS, d_hi);
        if constexpr (P2) store_row(LY::OFF_DS + PS_BYTES, d_lo);
      }
      if constexpr (P2) {
        if (j > 0 && j % FLUSH == 0 && mine) {         // (every product so far is done, and the next ones wait for this step's P)
          ptx::tc_fence_after();
          take_sums();
        }
      }
      ptx::fence_proxy_async_smem();
      ptx::tc_fence_before();
      ptx::mbar_arrive(bar(PDS_FULL + buf));
      if constexpr (SEQ) {
        ok = wait_all(bar(DV_DONE + buf), ph);
        if (!ok) break;
        store_row(LY::OFF_DS, d_hi);
        store_row(LY::OFF_DS + PS_BYTES, d_lo);
        ptx::fence_proxy_async_smem();
        ptx::mbar_arrive(bar(DS_FULL + buf));
      }
    }
    // epilogue: dV^T, dK^T [d = TMEM lane][key = column] -> dV, dK [batch][key][KV head][d]; one warpgroup each
    const int n_done = ok ? *reinterpret_cast<volatile int*>(&misc->total) : 0;
    if (ok && n_done > 0) ok = wait_all(bar(ACC_DONE + (n_done - 1) % NST), (uint32_t)((n_done - 1) / NST) & 1u);
    if (ok && mine && (n_done > 0 || a.n_split == 1)) {
      ptx::tc_fence_after();
      const int d = HD == 128 ? m : m & 63;
      float* out = (wg == 0 ? a.dV : a.dK) + (((long long)b * dm.seq_kv + k0) * dm.h_kv + r) * HD + d;
      const float mul = wg == 0 ? 1.f : dm.sm_scale;
      const long long pitch = (long long)dm.h_kv * HD;
      auto put = [&](int key, float x) {
        if (k0 + key >= dm.seq_kv) return;
        if (a.n_split > 1) atomicAdd(out + key * pitch, x * mul); else out[key * pitch] = x * mul;
      };
      if constexpr (P2) {
        if (n_done > 0) take_sums();
#pragma unroll
        for (int cc = 0; cc < NKV; ++cc) put(cc, sums[cc]);
      } else {
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
          uint32_t v[32];
          if (n_done > 0) {
            DASH_TMEM_LD32(v, sum_addr + half * 32);
            ptx::tmem_wait_ld();
          } else {
#pragma unroll
            for (int cc = 0; cc < 32; ++cc) v[cc] = 0u;
          }
#pragma unroll
          for (int cc = 0; cc < 32; ++cc) put(half * 32 + cc, __uint_as_float(v[cc]));
        }
      }
    }
    ptx::tc_fence_before();
  }

  __syncthreads();
  if (warp == W_SD) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, TMEM_COLS);
  }
  if (misc->abort_flag) {
    for (int k = tid; k < NKV * HD; k += THREADS) {
      const int key = k0 + k / HD;
      const long long at = (((long long)b * dm.seq_kv + key) * dm.h_kv + r) * HD + k % HD;
      if (key < dm.seq_kv) a.dK[at] = a.dV[at] = gave_up();      // (what other blocks add to it does not change it)
    }
  }
  if (tid == 0 && misc->abort_flag) report_error(a.sb, DASH_ERR_TIMEOUT, 121);
}

}  // namespace dkv

// [batch, tokens, heads, hd] bf16 tensor with element strides s[3]; box = 64 x box_heads x box_tokens x 1.
bool make_map(CUtensorMap* out, const void* base, int hd, long long tokens, int heads, int batch, const long long* s,
              int box_heads, int box_tokens) {
  cuuint64_t dims[4] = {(cuuint64_t)hd, (cuuint64_t)heads, (cuuint64_t)tokens, (cuuint64_t)batch};
  auto st = [](long long e) { return (cuuint64_t)((e > 0 ? e : 8) * 2); };
  cuuint64_t strides[3] = {st(s[2]), st(s[1]), st(s[0])};
  cuuint32_t box[4] = {64u, (cuuint32_t)box_heads, (cuuint32_t)box_tokens, 1u};
  return encode_bf16_sw128_4d(out, base, dims, strides, box);
}

// dK / dV, then dQ / dbias (which overwrites what the first one reads: see the top of the file)
template <int HD, int CPS, int WT, bool P2>
cudaError_t launch_kernels(const BwdArgs& a, const BwdMaps& m, cudaStream_t st) {
  const long long groups = (long long)a.dm.batch * a.dm.h_kv;
  constexpr int MTQ = 32 * (WT > 0 ? WT : 2), TPL = WT > 2 ? 4 : 2;
  cudaError_t e;
  {
    auto kern = dkv::attend_bwd_dkv_kernel<HD, CPS, TPL, P2>;
    constexpr uint32_t smem = dkv::Layout<HD, CPS, 32 * TPL, P2>::SMEM;
    static std::atomic<unsigned long long> configured{0};
    if ((e = allow_dynamic_smem(kern, smem, configured)) != cudaSuccess) return e;
    e = launch_chained(kern, dim3((unsigned)(a.n_slices * groups), a.n_split), dim3(dkv::threads(P2)), smem, st, m.qr, m.gr, m.k, m.v, a);
    count_launch();
    if (e != cudaSuccess) return e;
  }
  auto kern = dq::attend_bwd_dq_kernel<HD, CPS, WT, P2>;
  constexpr uint32_t smem = dq::Layout<HD, CPS, MTQ>::SMEM;
  static std::atomic<unsigned long long> configured{0};
  if ((e = allow_dynamic_smem(kern, smem, configured)) != cudaSuccess) return e;
  e = launch_chained(kern, dim3((unsigned)(a.n_tiles * groups)), dim3(dq::THREADS), smem, st, m.q, m.g, m.kc, m.vc, a);
  count_launch();
  return e;
}

template <int HD, int CPS>
cudaError_t launch_two_term(const BwdArgs& a, const BwdMaps& m, cudaStream_t st) {
  if (a.dm.g_q == 1) return launch_kernels<HD, CPS, 4, true>(a, m, st);
  if constexpr (CPS > 1) {
    if (a.TQ > a.dm.B) return launch_kernels<HD, CPS, 2, true>(a, m, st);
  }
  return launch_kernels<HD, CPS, 0, true>(a, m, st);
}

}  // namespace

bool prefill_bwd_sm100_supported(const Dims& dm) {
  if (!prefill_sm100_supported(dm) || broadcasts(dm.os, dm.batch, dm.seq_q, dm.h_q)) return false;      // (os: dO)
  return dm.qs[2] % 8 == 0 && dm.qs[1] % 8 == 0;      // 16-byte stores of dQ rows
}

cudaError_t launch_attend_prefill_bwd_sm100(const Dims& dm, bool two_term, int n_sm, const void* Q, const void* K, const void* V,
                                            const void* dO, const uint32_t* mask, const float* blk_bias, void* dQ, float* dK,
                                            float* dV, float* dbias, StatusBlock* sb, cudaStream_t st) {
  BwdArgs a;
  a.dm = dm;
  a.TQ = 128 / dm.g_q;
  a.n_tiles = (dm.seq_q + a.TQ - 1) / a.TQ;
  a.n_slices = (dm.seq_kv + NKV - 1) / NKV;
  a.inject = test_hooks().skip_own_k_load;
  a.wait_limit = test_hooks().wait_limit_cycles;
  a.Q = (const __nv_bfloat16*)Q; a.dO = (const __nv_bfloat16*)dO;
  a.mask = mask; a.blk_bias = blk_bias; a.marks = reinterpret_cast<int*>(dbias);
  a.dQ = (__nv_bfloat16*)dQ; a.dK = dK; a.dV = dV; a.dbias = dbias; a.sb = sb;
  // a row's statistics at the start of its dQ row
  a.stats.base = reinterpret_cast<char*>(dQ);
  a.stats.sb = dm.qs[0] * 2; a.stats.si = dm.qs[1] * 2; a.stats.sh = dm.qs[2] * 2; a.stats.sr = a.stats.sh * dm.g_q;
  // A slice's walk is a chain of one tile after another (one block per SM).  Where the slices alone leave SMs idle, several
  // blocks share a slice's tiles and add their sums with atomics; with one bf16 term dK and dV keep one owner per element.
  a.n_split = 1;
  cudaError_t e = cudaSuccess;
  if (two_term) {
    const long long blocks = (long long)a.n_slices * dm.batch * dm.h_kv;
    a.n_split = (int)std::max<long long>(1, std::min<long long>({2 * n_sm / blocks, a.n_tiles / 4, 16}));
  }
  BwdMaps m;
  const int box_kv = dm.B < NKV ? dm.B : NKV;
  if (!make_map(&m.q, Q, dm.d, dm.seq_q, dm.h_q, dm.batch, dm.qs, dm.g_q, a.TQ)) return cudaErrorInvalidValue;
  if (!make_map(&m.g, dO, dm.d, dm.seq_q, dm.h_q, dm.batch, dm.os, dm.g_q, a.TQ)) return cudaErrorInvalidValue;
  // (a run of the dK / dV kernel has at most 32 tokens)
  if (!make_map(&m.qr, Q, dm.d, dm.seq_q, dm.h_q, dm.batch, dm.qs, dm.g_q, std::min(a.TQ, 32))) return cudaErrorInvalidValue;
  if (!make_map(&m.gr, dO, dm.d, dm.seq_q, dm.h_q, dm.batch, dm.os, dm.g_q, std::min(a.TQ, 32))) return cudaErrorInvalidValue;
  if (!make_map(&m.k, K, dm.d, dm.seq_kv, dm.h_kv, dm.batch, dm.ks, 1, NKV)) return cudaErrorInvalidValue;
  if (!make_map(&m.v, V, dm.d, dm.seq_kv, dm.h_kv, dm.batch, dm.vs, 1, NKV)) return cudaErrorInvalidValue;
  if (!make_map(&m.kc, K, dm.d, dm.seq_kv, dm.h_kv, dm.batch, dm.ks, 1, box_kv)) return cudaErrorInvalidValue;
  if (!make_map(&m.vc, V, dm.d, dm.seq_kv, dm.h_kv, dm.batch, dm.vs, 1, box_kv)) return cudaErrorInvalidValue;
  if ((e = launch_attend_bwd_stats(a, m, st)) != cudaSuccess) return e;
  const long long rows = (long long)dm.batch * dm.h_kv * dm.seq_q;
  e = launch_chained(list_marks_kernel, dim3((unsigned)((rows + 255) / 256)), dim3(256), 0, st, dm, mask, a.marks, dK, dV,
                     a.n_split > 1 ? (long long)dm.batch * dm.seq_kv * dm.h_kv * dm.d : 0LL);
  count_launch();
  if (e != cudaSuccess) return e;

  if (!two_term) {
    if (dm.d != 128 || dm.B < NKV || dm.g_q < 2) return cudaErrorInvalidValue;
    return launch_kernels<128, 1, 0, false>(a, m, st);
  }
  if (dm.d == 128)
    return dm.B >= NKV ? launch_two_term<128, 1>(a, m, st) : dm.B == 32 ? launch_two_term<128, 2>(a, m, st) : launch_two_term<128, 4>(a, m, st);
  return dm.B >= NKV ? launch_two_term<64, 1>(a, m, st) : dm.B == 32 ? launch_two_term<64, 2>(a, m, st) : launch_two_term<64, 4>(a, m, st);
}

}  // namespace dash
