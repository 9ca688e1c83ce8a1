// Stage 2, decode, on TMA + tcgen05 for sm_100a (Eq. 7 / Proposition 1; Algorithm 3; split-KV of Section 3.5).
//
// HBM-bound: per (batch, KV head) only the routed chunks' K and V rows are read, once, by bulk tensor
// copies into a shared-memory ring of three 32 KiB tiles (K and V of a step of 128 KV tokens in turn), two blocks per SM,
// so enough bytes are in flight to cover DRAM latency without occupying threads, and one block's set-up and partial
// results pass under the other one's stream.  The arithmetic is tiny (g_q <= 16 query rows per KV
// head) and rides on the tensor cores in "transposed" form so that the KV tokens fill the MMA's M:
//     S^T[128 keys x 16 heads] = K_tile[128 x d] * Q^T[d x 16]          (heads padded to N = 16)
//     O^T[d = 128 x 16 heads] += V_tile^T[128 x 128 keys] * P^T[128 keys x 16]
// One softmax thread per key row (= TMEM lane of S^T); the per-head running maximum is shared through a
// small shared-memory reduction, the accumulator O^T is only 16 TMEM columns, so rescaling it is cheap.
// P enters its product as two bf16 terms (hi + lo, 16 bits of mantissa): with one, the weight of a split's own maximum was the
// only exact one, so every change of the split count moved the output by 2e-3, and fewer splits meant a larger error
// (48 paged caches, against float64: 2.07e-3 in up to 16 splits, 2.10e-3 in as few as the lists need, 1.66e-3 = the rounding
// of the output now).  Up to eight heads leave half of the MMA's N = 16 free: the lo terms take it, at no further product.
// The routed list (plus the row's own, possibly partial, chunk) is cut into n_split contiguous ranges of
// 64-token sub-blocks, one thread block each; the block that sees the last arrival of its (batch, KV head)
// merges the partial (m, l, O) of all splits in split order (or, without a workspace, a separate merge kernel does).
// Every wait on an mbarrier is bounded (DASH_ERR_TIMEOUT in the status word).  The fused step's cluster barriers have no limit
// and need none: every thread of a cluster reaches all of them, also after a wait of its block has run out.
//
// FUSED: the whole decode step in one launch, a cluster of CS blocks per (batch, KV head), where the grid is at most
// two blocks per SM and caches have up to 512 chunks: such a step is launches and round trips to L2.  Each block scores its share of
// the candidates and hands its logits to all of them through distributed shared memory, every block routes the group for
// itself (decode_route.cuh) and attends its share of the list, and the partial results meet through distributed shared memory
// as well.  One 8K cache, 8 KV heads: 13.4 us as routing and attention kernels, 9.3 fused.
#pragma once
#include <cuda.h>

#include "decode_route.cuh"
#include "sm100_ptx.cuh"
#include "tensor_map.cuh"

namespace dash {

struct DecodeArgs {
  Dims dm;
  const float* Kbar;     // FUSED only
  int n_split;
  int resident, least;   // blocks that are resident at once; sub-blocks a split has at least, where a group may use fewer splits than the grid has (0: it may not)
  const int* kv_len;
  const int* count;
  const int* blk_idx;
  const float* blk_bias;
  const __nv_bfloat16* Q;
  float* partials;
  __nv_bfloat16* O;      // non-null: fused merge by the last split of each (batch, KV head)
  StatusBlock* sb;
};

namespace {

constexpr int HD_MAX = 128;             // the shared-memory layout is the one of head_dim 128 (head_dim 64 fills half a tile)
constexpr int SUB = 64;                 // KV tokens per sub-block (one TMA box pair)
constexpr int STEP = 128;               // KV tokens per step = MMA M
constexpr int NSL = 3;                  // ring of K and V tiles: tile 2j = K of step j, 2j + 1 = its V
constexpr int NH = 16;                  // heads padded to the MMA N
constexpr int DEC_THREADS = 192;
// sub-blocks one thread block can own (a second tile of P terms leaves less room for their list)
__host__ __device__ constexpr int max_range(int g) { return g > 8 ? 288 : 512; }
constexpr uint32_t TILE_BYTES = STEP * HD_MAX * 2;   // 32 KiB: two regions (d halves) of 128 rows x 128 B
constexpr uint32_t QT_BYTES = NH * HD_MAX * 2;       // 4 KiB: two regions of 16 rows x 128 B
constexpr uint32_t PT_BYTES = NH * STEP * 2;     // 4 KiB: two regions (key halves) of 16 rows x 128 B
constexpr uint32_t OFF_KV = 0;
constexpr uint32_t OFF_QT = OFF_KV + NSL * TILE_BYTES;
constexpr uint32_t OFF_PT = OFF_QT + QT_BYTES;
__host__ __device__ constexpr uint32_t off_misc(int g) { return OFF_PT + (g > 8 ? 2 : 1) * PT_BYTES; }     // the lo terms: rows 8 .. 15 of P^T, or a tile of their own
constexpr uint32_t TMEM_COLS = 64;      // S^T buffers at columns 0 and 16, O^T at 32
enum BarD { Q_READY = 0, S_FULL = 1, P_FULL = 3, P_EMPTY = 5, RED_BAR = 6, LRED_BAR = 8, FULL = 9, EMPTY = 9 + NSL, N_BARS = 9 + 2 * NSL };
// CPS = routed chunks per 64-token sub-block: 1 for chunks of 64 / 128 tokens, 2 / 4 for chunks of 32 / 16 (a
// sub-block then gathers that many chunks of the list, each fetched by its own TMA box and carrying its own bias).
template <int CPS, int G>
struct MiscT {
  static constexpr int RANGE = max_range(G) / CPS;   // sub-blocks one thread block can own
  unsigned long long bar[N_BARS];
  uint32_t tmem_base;
  int abort_flag;
  float bias2[NSL][2][CPS];   // of the step whose V tile is in the slot
  int nvalid[NSL][2];
  float red[2][4][NH];
  float lred[4][NH];
  int is_last;               // this block saw the last arrival of its (batch, KV head); FUSED: length of the list
  int idx_s[RANGE][CPS];     // first KV token of each chunk slot of each owned sub-block (paged cache: inside its page)
  int pg_s[RANGE][CPS];      // outermost TMA coordinate of the slot: the sequence, or the physical page
  float bias_s[RANGE][CPS];
  unsigned short nval_s[RANGE];   // valid rows of the sub-block
};
template <int CPS, int G>
constexpr uint32_t dec_smem() {
  constexpr uint32_t bytes = off_misc(G) + (uint32_t)sizeof(MiscT<CPS, G>);
  static_assert(bytes <= 115712, "two blocks per SM");
  return bytes;
}

// FUSED: most chunks of a cache, and where the logits, the lists and (after the walk) the partial results
// sit in the ring of tiles
constexpr int FUSED_MAX_CHUNKS = 512;
constexpr uint32_t OFF_LIST = OFF_KV + 2 * TILE_BYTES;
struct ListS {
  int chunk[FUSED_MAX_CHUNKS];
  float bias[FUSED_MAX_CHUNKS];
  float taus[32], wsum[32];
  int wcnt[33];
};
static_assert(NH * (FUSED_MAX_CHUNKS + 64) * 4 <= 2 * TILE_BYTES && sizeof(ListS) <= TILE_BYTES, "logits and lists fit the ring");


__device__ __forceinline__ void tmem_ld16(uint32_t* r, uint32_t addr) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                 "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t addr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
               ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                 "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
               : "memory");
}

// head_dim 64 (HD = 64): K and V tiles are one 128-byte region per row.  S^T = K Q^T has four K steps.  The
// accumulator O^T would have only 64 rows, which is not an M = 128 shape, so the two 64-key sub-blocks of a step are
// stacked along M instead: A = [V_a^T ; V_b^T] (two MN blocks of 64, 8 KiB apart), K = 64 keys, B = [P_a^T | P_b^T]
// (N = 32): rows 0-63 / columns 0-15 hold V_a^T P_a^T and rows 64-127 / columns 16-31 hold V_b^T P_b^T (the other two
// quadrants are not used); the two are added when the partial is written.
// CS: blocks per cluster (FUSED), 0: attention alone.
template <int G, int CPS, int HD, int CS>
__global__ void __launch_bounds__(DEC_THREADS, 2)
decode_sm100_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, DecodeArgs a) {
  constexpr bool FUSED = CS > 0;
  constexpr int NC = FUSED ? CS : 1;
  using MiscD = MiscT<CPS, G>;
  constexpr int W = SUB / CPS;          // rows of one chunk slot inside a sub-block
  extern __shared__ __align__(1024) uint8_t smem[];
  MiscD* misc = reinterpret_cast<MiscD*>(smem + off_misc(G));
  const Dims& dm = a.dm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t sbase = ptx::smem_u32(smem);
  auto bar = [&](int i) { return ptx::smem_u32(&misc->bar[i]); };
  volatile int* abort_flag = &misc->abort_flag;
  const int split = blockIdx.x, r = blockIdx.y, b = blockIdx.z;
  int n_split = FUSED ? NC : a.n_split;      // (a cluster is the blocks of one group: split = rank)

  // A block of a short list lives for a few round trips to memory, so independent ones start together: the descriptors here,
  // the lengths of sequence and list and the status word behind the wait.
  warm_length(a.kv_len, b);
  const long long grp = (long long)b * dm.h_kv + r;
  const int spb = CPS > 1 ? 1 : dm.B / SUB;                     // sub-blocks per routed chunk (chunks >= 64 tokens)
  int L = 0, c_own = 0, own_tokens = 0;                          // own_tokens: 1 .. B
  int n_routed = 0, n_routed_sub = 0, n_items = 0;
  auto read_lengths = [&]() {
    const int len = a.kv_len ? a.kv_len[b] : dm.seq_kv, status = a.sb ? *reinterpret_cast<volatile int*>(&a.sb->status) : 0;
    if constexpr (!FUSED) n_routed = a.count[grp];
    L = max(1, min(len, dm.seq_kv));
    c_own = (L - 1) >> dm.log_b;
    own_tokens = L - c_own * dm.B;
    return status;
  };
  auto list_size = [&]() {
    DASH_CHECK(n_routed >= 0 && n_routed <= min(c_own, dm.T_s), a.sb, 310, n_routed = 0);
    n_routed_sub = CPS > 1 ? (n_routed + CPS - 1) / CPS : n_routed * spb;
    n_items = n_routed_sub + (own_tokens + SUB - 1) / SUB;
  };
  // A short list takes fewer splits than the grid has: a block costs about six sub-blocks of streaming beside its share
  // (48 paged sequences of 1K to 32K, lists of 20 chunks on average and up to 128).  A surplus block leaves at once, one that
  // is not among the first before it has set anything up.
  bool waited = false;
  int status = 0;
  if constexpr (!FUSED) {
    if ((long long)blockIdx.x + (long long)gridDim.x * (blockIdx.y + (long long)gridDim.y * blockIdx.z) >= a.resident) {
      chain_wait();
      waited = true;
      status = read_lengths();
      list_size();
      if (a.least > 0) n_split = max(1, min(n_split, n_items / a.least));
      if (split >= n_split) return;
    }
  }
  if (tid == 128) {
    ptx::prefetch_tensormap(&tmK);
    ptx::prefetch_tensormap(&tmV);
  }
  if (tid == 0) {
    misc->abort_flag = 0;
    if ((sbase & 1023u) != 0u) {
      report_error(a.sb, DASH_ERR_CUDA, 300);
      misc->abort_flag = 1;
    }
    ptx::mbar_init(bar(Q_READY), 128);
    ptx::mbar_init(bar(S_FULL), 1);
    ptx::mbar_init(bar(S_FULL + 1), 1);
    ptx::mbar_init(bar(P_FULL), 128);
    ptx::mbar_init(bar(P_FULL + 1), 128);
    ptx::mbar_init(bar(P_EMPTY), 1);
    ptx::mbar_init(bar(RED_BAR), 128);
    ptx::mbar_init(bar(RED_BAR + 1), 128);
    ptx::mbar_init(bar(LRED_BAR), 128);
    for (int s = 0; s < NSL; ++s) {
      ptx::mbar_init(bar(FULL + s), 1);
      ptx::mbar_init(bar(EMPTY + s), 1);
    }
    ptx::fence_barrier_init();
  }
  if (warp == 5) {
    ptx::tmem_alloc(ptx::smem_u32(&misc->tmem_base), TMEM_COLS);
    ptx::tmem_relinquish();
    ptx::tc_fence_before();
  }
  __syncthreads();
  if constexpr (FUSED) ptx::cluster_sync_all();      // every block runs before anybody writes into its shared memory
  ptx::tc_fence_after();
  const uint32_t tmem = misc->tmem_base;

  // barriers and tensor memory are set up; everything below reads what the routing kernels wrote
  if (!waited) {
    chain_wait();
    status = read_lengths();
  }
  // an error already in the status word makes every role leave at its first wait (see the prefill kernel)
  if (status != 0) *abort_flag = 1;
  __syncthreads();
  ListS* list = reinterpret_cast<ListS*>(smem + OFF_LIST);
  if constexpr (FUSED) {
    const int n_vis = min(c_own, dm.T_s), n_cand = max(n_vis - dm.local_blocks, 0);
    const int stride = route_stride(n_vis), share = (n_cand + NC - 1) / NC;
    float* X = reinterpret_cast<float*>(smem + OFF_KV);       // [G][stride]
    if (split * share < n_cand) {
      float q[G][HD / 32];
      load_query<__nv_bfloat16, HD, G>(dm, a.Q, b, r, lane, q);
      const float* kb = a.Kbar + grp * dm.T_s * HD + lane * (HD / 32);
      score_rows<HD, G>(q, kb, split * share, min(n_cand, (split + 1) * share), warp, DEC_THREADS / 32, lane, [&](int g, int c, float x) {
        const uint32_t at = sbase + OFF_KV + (uint32_t)(g * stride + c) * 4;
#pragma unroll
        for (int k = 0; k < NC; ++k) ptx::st_cluster_f32(ptx::map_to_rank(at, k), x);
      });
    }
    __syncwarp();
    ptx::cluster_sync_all();
    route_group<G, DEC_THREADS / 32, 16>(
        dm, X, stride, n_cand, n_vis, (n_vis + 31) / 32, list->taus, list->wsum, list->wcnt, warp, lane, [](int, uint32_t) {},
        [&](int n) { if (tid == 0) misc->is_last = n; }, [&](int pos, int c, float bias) { list->chunk[pos] = c; list->bias[pos] = bias; });
    ptx::fence_proxy_async_smem();       // the ring is TMA's from here on
    __syncthreads();
    n_routed = misc->is_last;            // (not in the ring: the producer may already be refilling that)
  }
  if (!waited) {
    list_size();
    if constexpr (!FUSED) {
      if (a.least > 0) n_split = max(1, min(n_split, n_items / a.least));
      if (split >= n_split) {
        if (warp == 5) {
          ptx::tc_fence_after();
          ptx::tmem_dealloc(tmem, TMEM_COLS);
        }
        return;
      }
    }
  }
  const int per = (n_items + n_split - 1) / n_split;
  const int lo = min(n_items, split * per), hi = min(n_items, lo + per);
  const int n_own = hi - lo;                                     // <= max_range(G) by the host's choice of n_split
  const int n_steps = (n_own + 1) / 2;

  const long long loff = grp * dm.list_rows;

  if (warp == 4) {
    // ---------------- producer
    // owned sub-blocks -> (first token, bias, valid rows), staged once so the walk has no dependent global reads
    for (int k = lane; k < n_own; k += 32) {
      const int it = lo + k;
      if constexpr (CPS > 1) {
        if (it < n_routed_sub) {
          // CPS consecutive list entries; a short last group repeats its last chunk in rows that are marked invalid
          const int e0 = it * CPS, m = min(CPS, n_routed - e0);
#pragma unroll
          for (int s = 0; s < CPS; ++s) {
            const int e = e0 + min(s, m - 1);
            int cc = FUSED ? list->chunk[e] : a.blk_idx[loff + e];
            DASH_CHECK(cc >= 0 && cc < c_own, a.sb, 311, cc = 0);
            kv_locate(dm, b, cc * dm.B, &misc->pg_s[k][s], &misc->idx_s[k][s]);
            DASH_CHECK(!dm.page_table || (unsigned)misc->pg_s[k][s] < (unsigned)dm.num_pages, a.sb, 313, misc->pg_s[k][s] = 0);
            misc->bias_s[k][s] = FUSED ? list->bias[e] : a.blk_bias[loff + e];
          }
          misc->nval_s[k] = (unsigned short)(m * dm.B);
        } else {
          // the own chunk (shorter than a sub-block) repeats in every slot, all but the first marked invalid: the chunk behind it
          // may lie in a page that the table does not hold
          int pg, tok;
          kv_locate(dm, b, c_own * dm.B, &pg, &tok);
          DASH_CHECK(!dm.page_table || (unsigned)pg < (unsigned)dm.num_pages, a.sb, 315, pg = 0);
#pragma unroll
          for (int s = 0; s < CPS; ++s) {
            misc->pg_s[k][s] = pg;
            misc->idx_s[k][s] = tok;
            misc->bias_s[k][s] = 0.f;
          }
          misc->nval_s[k] = (unsigned short)(L - c_own * dm.B);
        }
        continue;
      }
      int tok0, nv;
      float bs;
      if (it < n_routed_sub) {
        const int e = it / spb, sub = it % spb;
        int cc = FUSED ? list->chunk[e] : a.blk_idx[loff + e];
        DASH_CHECK(cc >= 0 && cc < c_own, a.sb, 312, cc = 0);
        tok0 = cc * dm.B + sub * SUB;
        bs = FUSED ? list->bias[e] : a.blk_bias[loff + e];
        nv = SUB;
      } else {
        const int sub = it - n_routed_sub;
        tok0 = c_own * dm.B + sub * SUB;
        bs = 0.f;
        nv = min(SUB, L - tok0);
      }
      kv_locate(dm, b, tok0, &misc->pg_s[k][0], &misc->idx_s[k][0]);
      DASH_CHECK(!dm.page_table || (unsigned)misc->pg_s[k][0] < (unsigned)dm.num_pages, a.sb, 314, misc->pg_s[k][0] = 0);
      misc->bias_s[k][0] = bs; misc->nval_s[k] = (unsigned short)nv;
    }
    __syncwarp();
    if (lane == 0) {
      bool ok = true;
      int s = 0, ph = 1;
      for (int j = 0; j < n_steps && ok; ++j) {
        const int k0 = 2 * j, k1 = (2 * j + 1 < n_own) ? 2 * j + 1 : 2 * j;   // an odd tail repeats its last sub-block
        // one 128-row tile: sub-blocks k0 and k1, each CPS boxes of W rows, for both halves of head_dim
        auto load_tile = [&](const CUtensorMap* tm, uint32_t dst, uint32_t barrier) {
          ptx::mbar_arrive_expect_tx(barrier, STEP * HD * 2);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int k = h ? k1 : k0;
#pragma unroll
            for (int q = 0; q < CPS; ++q) {
              const int tok = misc->idx_s[k][q], pg = misc->pg_s[k][q];
              const uint32_t d = dst + (h * SUB + q * W) * 128;
              ptx::tma_load_4d(d, tm, barrier, 0, r, tok, pg);
              if constexpr (HD == 128) ptx::tma_load_4d(d + TILE_BYTES / 2, tm, barrier, 64, r, tok, pg);
            }
          }
        };
        auto advance = [&]() { if (++s == NSL) { s = 0; ph ^= 1; } };
        ok = ptx::mbar_wait(bar(EMPTY + s), ph, abort_flag);
        if (!ok) break;
        load_tile(&tmK, sbase + OFF_KV + s * TILE_BYTES, bar(FULL + s));
        advance();
        ok = ptx::mbar_wait(bar(EMPTY + s), ph, abort_flag);
        if (!ok) break;
#pragma unroll
        for (int q = 0; q < CPS; ++q) {
          misc->bias2[s][0][q] = misc->bias_s[k0][q];
          misc->bias2[s][1][q] = misc->bias_s[k1][q];
        }
        misc->nvalid[s][0] = misc->nval_s[k0];
        misc->nvalid[s][1] = (k1 != k0) ? misc->nval_s[k1] : 0;
        load_tile(&tmV, sbase + OFF_KV + s * TILE_BYTES, bar(FULL + s));
        advance();
      }
      if (!ok) {
        for (int q = 0; q < NSL; ++q)
          for (int k = 0; k < 200000 && !ptx::mbar_try_wait(bar(FULL + q), 0) && !ptx::mbar_try_wait(bar(FULL + q), 1); ++k) {}
      }
    }
  } else if (warp == 5) {
    // ---------------- MMA issuer
    if (lane == 0 && n_steps > 0) {
      constexpr uint32_t IDESC_S = ptx::idesc_bf16_f32(128, NH, false, false);
      constexpr uint32_t IDESC_O = ptx::idesc_bf16_f32(128, HD == 128 ? NH : 2 * NH, true, false);
      const uint64_t kd0 = ptx::smem_desc_sw128(sbase + OFF_KV, 16, 1024);
      const uint64_t qd0 = ptx::smem_desc_sw128(sbase + OFF_QT, 16, 1024);
      // MN-major A: the two MN blocks of 64 are the d halves, 16 KiB apart (head_dim 128), or the two 64-key
      // sub-blocks of the step, 8 KiB apart (head_dim 64)
      const uint64_t vd0 = ptx::smem_desc_sw128(sbase + OFF_KV, HD == 128 ? TILE_BYTES / 2 : SUB * 128, 1024);
      const uint64_t pd0 = ptx::smem_desc_sw128(sbase + OFF_PT, 16, 1024);
      bool ok = ptx::mbar_wait(bar(Q_READY), 0, abort_flag);
      // tile 2j (K) and 2j + 1 (V) of the ring
      int ks = 0, kph = 0, vs = 1, vph = 0;
      auto next_step = [](int& slot, int& phase) { slot += 2; if (slot >= NSL) { slot -= NSL; phase ^= 1; } };
      auto issue_s = [&](int j) -> bool {
        if (!ptx::mbar_wait(bar(FULL + ks), kph, abort_flag)) return false;
        ptx::tc_fence_after();
        const uint64_t kd = kd0 + (uint64_t)((ks * TILE_BYTES) >> 4);
#pragma unroll
        for (int k = 0; k < HD / 16; ++k) {
          const uint64_t ad = kd + (uint64_t)(((k >> 2) * (TILE_BYTES / 2) + (k & 3) * 32) >> 4);
          const uint64_t bd = qd0 + (uint64_t)(((k >> 2) * (QT_BYTES / 2) + (k & 3) * 32) >> 4);
          ptx::mma_bf16_ss(tmem + (j & 1) * NH, ad, bd, IDESC_S, k > 0 ? 1u : 0u);
        }
        ptx::mma_commit(bar(S_FULL + (j & 1)));
        ptx::mma_commit(bar(EMPTY + ks));
        next_step(ks, kph);
        return true;
      };
      if (ok) ok = issue_s(0);
      for (int j = 0; j < n_steps && ok; ++j) {
        if (j + 1 < n_steps) ok = issue_s(j + 1);
        if (!ok) break;
        ok = ptx::mbar_wait(bar(FULL + vs), vph, abort_flag) && ptx::mbar_wait(bar(P_FULL + (j & 1)), (j >> 1) & 1, abort_flag);
        if (!ok) break;
        ptx::tc_fence_after();
        const uint64_t vd = vd0 + (uint64_t)((vs * TILE_BYTES) >> 4);
#pragma unroll
        for (int k = 0; k < (HD == 128 ? STEP : SUB) / 16; ++k) {
          const uint64_t ad = vd + (uint64_t)((k * 16 * 128) >> 4);                                   // 16 key rows = 2048 B
          // head_dim 128: P^T is two K-major regions (key halves) of 16 rows; head_dim 64: the same bytes read as one
          // region of 32 rows (sub-block a's heads, then sub-block b's), 64 keys long
          const uint64_t bd = pd0 + (uint64_t)(((HD == 128 ? (k >> 2) * (PT_BYTES / 2) : 0) + (k & 3) * 32) >> 4);
          ptx::mma_bf16_ss(tmem + 2 * NH, ad, bd, IDESC_O, (j > 0 || k > 0) ? 1u : 0u);
          if constexpr (G > 8) ptx::mma_bf16_ss(tmem + 2 * NH, ad, bd + (uint64_t)(PT_BYTES >> 4), IDESC_O, 1u);     // the lo terms
        }
        ptx::mma_commit(bar(EMPTY + vs));
        ptx::mma_commit(bar(P_EMPTY));
        next_step(vs, vph);
      }
    }
    __syncwarp();
  } else {
    // ---------------- softmax: thread = key row of the step = TMEM lane of S^T; also lane d of O^T
    const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
    const float c1 = dm.sm_scale * 1.4426950408889634f;
    // Q^T tile: 16 rows (heads, zero beyond G) x 128 d, K-major, 128-byte swizzle; P^T rows of no head stay zero
    for (int ch = tid; ch < NH * 16; ch += 128) {
      const int h = ch >> 4, c16 = ch & 15;            // 16-byte chunk c16 of head h: d = c16*8 .. +7
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (h < G && c16 * 8 < HD)
        v = *reinterpret_cast<const uint4*>(a.Q + (long long)b * dm.qs[0] + (long long)(r * G + h) * dm.qs[2] + c16 * 8);
      const uint32_t off = (c16 >> 3) * (QT_BYTES / 2) + h * 128 + (((c16 & 7) ^ (h & 7)) << 4);
      *reinterpret_cast<uint4*>(smem + OFF_QT + off) = v;
      *reinterpret_cast<uint4*>(smem + OFF_PT + off) = make_uint4(0u, 0u, 0u, 0u);
    }
    ptx::fence_proxy_async_smem();
    ptx::mbar_arrive(bar(Q_READY));

    float m[G], l[G];
#pragma unroll
    for (int h = 0; h < G; ++h) { m[h] = -INFINITY; l[h] = 0.f; }
    const int half = tid >> 6, row = tid & 63;
    bool ok = true;
    int vs = 1, vph = 0;
    for (int j = 0; j < n_steps && ok; ++j) {
      ok = ptx::mbar_wait_warp(bar(FULL + vs), vph, abort_flag);     // step metadata visible, V tile landed
      if (!ok) break;
      const float b2 = misc->bias2[vs][half][CPS > 1 ? row / W : 0] * 1.4426950408889634f;
      const int nval = misc->nvalid[vs][half];
      const bool valid = row < nval;
      ok = ptx::mbar_wait_warp(bar(S_FULL + (j & 1)), (j >> 1) & 1, abort_flag);
      if (!ok) break;
      ptx::tc_fence_after();
      uint32_t sr[16];
      tmem_ld16(sr, lane_addr + (j & 1) * NH);
      ptx::tmem_wait_ld();
      float x[G];
#pragma unroll
      for (int h = 0; h < G; ++h) {
        x[h] = valid ? fmaf(__uint_as_float(sr[h]), c1, b2) : -INFINITY;
        const float wm = warp_max(x[h]);
        if (lane == 0) misc->red[j & 1][warp][h] = wm;
      }
      // per-head maxima of the four warps meet through shared memory (bounded mbarrier, not bar.sync)
      ptx::mbar_arrive(bar(RED_BAR + (j & 1)));
      ok = ptx::mbar_wait_warp(bar(RED_BAR + (j & 1)), (j >> 1) & 1, abort_flag);
      if (!ok) break;
      float corr[G];
      bool changed = false;
#pragma unroll
      for (int h = 0; h < G; ++h) {
        const float ms = fmaxf(fmaxf(misc->red[j & 1][0][h], misc->red[j & 1][1][h]),
                               fmaxf(misc->red[j & 1][2][h], misc->red[j & 1][3][h]));
        const float mn = fmaxf(m[h], ms);
        changed |= mn > m[h];
        corr[h] = exp2f(m[h] - mn);     // 0 while nothing has been accumulated
        m[h] = mn;
      }
      __nv_bfloat16 pb[G], pl[G];      // P = pb + pl
#pragma unroll
      for (int h = 0; h < G; ++h) {
        const float p = valid ? exp2f(x[h] - m[h]) : 0.f;
        l[h] = l[h] * corr[h] + p;
        pb[h] = __float2bfloat16_rn(p);
        pl[h] = __float2bfloat16_rn(p - __bfloat162float(pb[h]));
      }
      // the previous step's PV must be done before P^T is overwritten and before O^T is rescaled
      ok = ptx::mbar_wait_warp(bar(P_EMPTY), (j & 1) ^ 1, abort_flag);
      if (!ok) break;
      ptx::tc_fence_after();
      if (j > 0 && changed) {
        // head_dim 64: this lane's live accumulator columns are h (sub-block a, lanes 0-63) or NH + h (lanes 64-127)
        const uint32_t o_addr = lane_addr + 2 * NH + ((HD == 64 && half) ? NH : 0);
        uint32_t o[16];
        tmem_ld16(o, o_addr);
        ptx::tmem_wait_ld();
#pragma unroll
        for (int h = 0; h < G; ++h) {
          o[h] = __float_as_uint(__uint_as_float(o[h]) * corr[h]);
          if constexpr (G <= 8) o[8 + h] = __float_as_uint(__uint_as_float(o[8 + h]) * corr[h]);
        }
        tmem_st16(o_addr, o);
        ptx::tmem_wait_st();
      }
      // P^T[head h][key tid]: K-major rows of 64 keys, 128-byte swizzle
#pragma unroll
      for (int h = 0; h < G; ++h) {
        const uint32_t off = half * (PT_BYTES / 2) + h * 128 + ((((row >> 3) & 7) ^ (h & 7)) << 4) + (row & 7) * 2;
        *reinterpret_cast<__nv_bfloat16*>(smem + OFF_PT + off) = pb[h];
        *reinterpret_cast<__nv_bfloat16*>(smem + OFF_PT + off + (G <= 8 ? 8 * 128 : PT_BYTES)) = pl[h];      // (row 8 + h: the swizzle of row h)
      }
      // rows past the end of the sequence may hold anything (even NaN): zero their V rows, since 0 * NaN = NaN (also in the
      // half that repeats an odd tail's last sub-block, all of whose rows are invalid).  By the whole warp, a row's 16-byte
      // pieces in adjacent lanes: one row per lane would be 32 ways of bank conflict
      if (const int first = nval - (row & 32); first < 32) {      // this warp's rows from `first` on
        for (int q = max(first, 0) * 8 + lane; q < 32 * 8; q += 32) {
          uint8_t* piece = smem + OFF_KV + vs * TILE_BYTES + warp * (32 * 128) + q * 16;
          *reinterpret_cast<uint4*>(piece) = make_uint4(0u, 0u, 0u, 0u);
          if constexpr (HD == 128) *reinterpret_cast<uint4*>(piece + TILE_BYTES / 2) = make_uint4(0u, 0u, 0u, 0u);
        }
      }
      ptx::fence_proxy_async_smem();
      ptx::tc_fence_before();
      ptx::mbar_arrive(bar(P_FULL + (j & 1)));
      vs += 2;
      if (vs >= NSL) { vs -= NSL; vph ^= 1; }
    }

    // ---------------- partial (m, l, O) of this split
    if (ok && n_steps > 0) ok = ptx::mbar_wait_warp(bar(P_EMPTY), (n_steps - 1) & 1, abort_flag);
    ptx::tc_fence_after();
#pragma unroll
    for (int h = 0; h < G; ++h) {
      const float ls = warp_sum(l[h]);
      if (lane == 0) misc->lred[warp][h] = ls;
    }
    ptx::mbar_arrive(bar(LRED_BAR));
    ok = ptx::mbar_wait_warp(bar(LRED_BAR), 0, abort_flag) && ok;
    uint32_t o[16];
#pragma unroll
    for (int h = 0; h < 16; ++h) o[h] = 0u;
    if (ok && n_steps > 0) {
      tmem_ld16(o, lane_addr + 2 * NH + ((HD == 64 && (tid >> 6)) ? NH : 0));
      ptx::tmem_wait_ld();
    }
    if constexpr (G <= 8) {
#pragma unroll
      for (int h = 0; h < G; ++h) o[h] = __float_as_uint(__uint_as_float(o[h]) + __uint_as_float(o[8 + h]));
    }
    if constexpr (HD == 64) {
      // O^T[d][h] = (sub-block a's part in lane d) + (sub-block b's part in lane 64 + d): the upper lanes hand theirs
      // over through the P^T tile, which no product reads any more
      float* comb = reinterpret_cast<float*>(smem + OFF_PT);       // [64][16]
      if (tid >= 64) {
#pragma unroll
        for (int h = 0; h < G; ++h) comb[(tid - 64) * NH + h] = __uint_as_float(o[h]);
      }
      ptx::mbar_arrive(bar(LRED_BAR));
      ok = ptx::mbar_wait_warp(bar(LRED_BAR), 1, abort_flag) && ok;
      if (tid < 64) {
#pragma unroll
        for (int h = 0; h < G; ++h) o[h] = __float_as_uint(__uint_as_float(o[h]) + comb[tid * NH + h]);
      }
    }
    const int pitch = a.n_split;             // partial results of a head
    const long long pbase = (((long long)b * dm.h_q + (long long)r * G) * pitch + split) * (HD + 2);
#pragma unroll
    for (int h = 0; h < G; ++h) {
      // (m, l, O); FUSED: O, m, l in this block's own ring, whose tiles have all been consumed
      float* pp = FUSED ? reinterpret_cast<float*>(smem + OFF_KV) + h * (HD + 4) : a.partials + pbase + (long long)h * pitch * (HD + 2);
      if (tid < HD) pp[(FUSED ? 0 : 2) + tid] = (n_steps > 0) ? __uint_as_float(o[h]) : 0.f;   // thread tid holds O^T[d = tid][h]
      if (tid == h) {
        pp[FUSED ? HD : 0] = (n_steps > 0) ? m[h] * 0.6931471805599453f : -INFINITY;   // the merge works in natural-log units
        pp[FUSED ? HD + 1 : 1] = misc->lred[0][h] + misc->lred[1][h] + misc->lred[2][h] + misc->lred[3][h];
      }
    }
    if (!FUSED && n_split > 1) __threadfence();        // the partial is visible device-wide before this block counts itself as arrived
    ptx::tc_fence_before();
  }

  __syncthreads();
  // Not before: blocks of the next kernel that arrive while most of this grid still streams pile up on the SMs that were free
  // first, and stay there (3 caches of 104448 tokens with lists of 8 to 47 chunks: 31.4 us a step instead of 24).
  chain_release();
  if (warp == 5) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, TMEM_COLS);
  }
  if constexpr (FUSED) {
    // ---------------- rank k merges the heads k, k + NC, ... from all blocks' partial results, in rank order
    __syncwarp();
    ptx::cluster_sync_all();
    constexpr int VPL = HD / 32;
    for (int h = split + NC * warp; h < G; h += NC * (DEC_THREADS / 32)) {
      const uint32_t at = sbase + OFF_KV + (uint32_t)h * (HD + 4) * 4;
      const uint32_t mine = ptx::map_to_rank(at, lane & (NC - 1));
      const float ms = ptx::ld_cluster_f32(mine + HD * 4), ls = ptx::ld_cluster_f32(mine + HD * 4 + 4);
      float2 o[NC][VPL / 2];
#pragma unroll
      for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int v = 0; v < VPL / 2; ++v) o[k][v] = ptx::ld_cluster_f32x2(ptx::map_to_rank(at, k) + (lane * VPL + 2 * v) * 4);
      const float M = warp_max(ms);           // (by all lanes, whatever their split holds: a warp-wide instruction)
      const float w = ms > -INFINITY ? __expf(ms - M) : 0.f;
      const float Lsum = warp_sum(lane < NC ? w * ls : 0.f);
      float2 acc[VPL / 2];
#pragma unroll
      for (int v = 0; v < VPL / 2; ++v) acc[v] = make_float2(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const float wk = __shfl_sync(0xffffffffu, w, k);
#pragma unroll
        for (int v = 0; v < VPL / 2; ++v) { acc[v].x += wk * o[k][v].x; acc[v].y += wk * o[k][v].y; }
      }
      const float inv = Lsum > 0.f ? 1.f / Lsum : 0.f;
      __nv_bfloat16* op = a.O + (long long)b * dm.os[0] + (long long)(r * G + h) * dm.os[2] + lane * VPL;
#pragma unroll
      for (int v = 0; v < VPL / 2; ++v) {
        op[2 * v] = __float2bfloat16_rn(acc[v].x * inv);
        op[2 * v + 1] = __float2bfloat16_rn(acc[v].y * inv);
      }
    }
    __syncwarp();
    ptx::cluster_sync_all();      // nobody leaves while a peer may still read its shared memory
  } else if (a.O != nullptr) {
    // ---------------- the last split of this (batch, KV head) to arrive merges all of them, in split order
    int* counter = arrival_counters(a.sb) + grp;
    if (tid == 0) {
      const bool last = n_split == 1 || atomicAdd(counter, 1) == n_split - 1;
      if (last && n_split > 1) *counter = 0;          // every split has arrived: the counter is ready for the next launch
      misc->is_last = last ? 1 : 0;
    }
    __syncthreads();
    if (misc->is_last) {
      __threadfence();
      constexpr int VPL = HD / 32;
      for (int h = warp; h < G; h += DEC_THREADS / 32) {
        const long long bh = (long long)b * dm.h_q + (long long)r * G + h;
        const float* p = a.partials + bh * a.n_split * (HD + 2);
        // lane s holds the weight of split s (at most 32 splits); the partial outputs are summed in split order, eight
        // loads in flight (one after another they cost a round trip to L2 each: 3.5 us at 16 splits)
        const float ms = lane < n_split ? __ldcg(p + lane * (HD + 2)) : -INFINITY;
        const float ls = lane < n_split ? __ldcg(p + lane * (HD + 2) + 1) : 0.f;
        const float M = warp_max(ms);
        const float w = ms > -INFINITY ? __expf(ms - M) : 0.f;
        const float Lsum = warp_sum(w * ls);
        float acc[VPL];
#pragma unroll
        for (int v = 0; v < VPL; ++v) acc[v] = 0.f;
        for (int s0 = 0; s0 < n_split; s0 += 8) {
          float2 o[8][VPL / 2];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (s0 + u < n_split) {
              const float2* po = reinterpret_cast<const float2*>(p + (s0 + u) * (HD + 2) + 2 + lane * VPL);   // 8-byte aligned
#pragma unroll
              for (int v = 0; v < VPL / 2; ++v) o[u][v] = __ldcg(po + v);
            }
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const float wu = __shfl_sync(0xffffffffu, w, (s0 + u) & 31);
            if (s0 + u < n_split) {
#pragma unroll
              for (int v = 0; v < VPL / 2; ++v) { acc[2 * v] += wu * o[u][v].x; acc[2 * v + 1] += wu * o[u][v].y; }
            }
          }
        }
        const float inv = Lsum > 0.f ? 1.f / Lsum : 0.f;
        __nv_bfloat16* op = a.O + (long long)b * dm.os[0] + (long long)(r * G + h) * dm.os[2] + lane * VPL;
#pragma unroll
        for (int v = 0; v < VPL; ++v) op[v] = __float2bfloat16_rn(acc[v] * inv);
      }
    }
  }
  if (tid == 0 && misc->abort_flag) report_error(a.sb, DASH_ERR_TIMEOUT, 301);
}

bool make_kv_map(CUtensorMap* out, const void* base, const Dims& dm, const long long* s) {
  // contiguous cache: [batch][seq_kv] tokens; paged cache: [num_pages][page_size]
  cuuint64_t dims[4] = {(cuuint64_t)dm.d, (cuuint64_t)dm.h_kv, (cuuint64_t)(dm.page_table ? dm.page_size : dm.seq_kv),
                        (cuuint64_t)(dm.page_table ? dm.num_pages : dm.batch)};
  auto st = [](long long e) { return (cuuint64_t)((e > 0 ? e : 8) * 2); };
  cuuint64_t strides[3] = {st(s[2]), st(s[1]), st(s[0])};
  cuuint32_t box[4] = {64u, 1u, (cuuint32_t)(dm.B < SUB ? dm.B : SUB), 1u};   // chunks below 64 tokens: one box per chunk
  return encode_bf16_sw128_4d(out, base, dims, strides, box);
}

template <int G, int CPS, int HD, int CS>
static cudaError_t launch_one(const CUtensorMap& tk, const CUtensorMap& tv, const DecodeArgs& a, cudaStream_t st) {
  auto kern = decode_sm100_kernel<G, CPS, HD, CS>;
  static std::atomic<unsigned long long> configured{0};
  constexpr uint32_t smem = dec_smem<CPS, G>();
  if (cudaError_t e = allow_dynamic_smem(kern, smem, configured); e != cudaSuccess) return e;
  const dim3 grid(CS > 0 ? CS : a.n_split, a.dm.h_kv, a.dm.batch);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(DEC_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see launch_chained
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = CS > 0 ? CS : 1;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = CS > 0 ? 2 : 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kern, tk, tv, a);
  count_launch();
  return e;
}

template <int CPS, int HD, int CS>
static cudaError_t launch_group_size(const CUtensorMap& tk, const CUtensorMap& tv, const DecodeArgs& a, cudaStream_t st) {
  switch (a.dm.g_q) {
    case 1: return launch_one<1, CPS, HD, CS>(tk, tv, a, st);
    case 2: return launch_one<2, CPS, HD, CS>(tk, tv, a, st);
    case 4: return launch_one<4, CPS, HD, CS>(tk, tv, a, st);
    case 8: return launch_one<8, CPS, HD, CS>(tk, tv, a, st);
    case 16: return launch_one<16, CPS, HD, CS>(tk, tv, a, st);
    default: return cudaErrorInvalidValue;
  }
}

template <int CS>
static cudaError_t launch_any(DecodeArgs& a, const void* K, const void* V, cudaStream_t st) {
  const Dims& dm = a.dm;
  CUtensorMap tk, tv;
  if (!make_kv_map(&tk, K, dm, dm.ks) || !make_kv_map(&tv, V, dm, dm.vs)) return cudaErrorInvalidValue;
  if (dm.d == 128)
    return dm.B >= SUB ? launch_group_size<1, 128, CS>(tk, tv, a, st) : dm.B == 32 ? launch_group_size<2, 128, CS>(tk, tv, a, st)
                                                                                     : launch_group_size<4, 128, CS>(tk, tv, a, st);
  return dm.B >= SUB ? launch_group_size<1, 64, CS>(tk, tv, a, st) : dm.B == 32 ? launch_group_size<2, 64, CS>(tk, tv, a, st)
                                                                                   : launch_group_size<4, 64, CS>(tk, tv, a, st);
}

}  // namespace

// One translation unit per cluster size (they compile in parallel).
cudaError_t launch_decode_cluster8(DecodeArgs& a, const void* K, const void* V, cudaStream_t st);
cudaError_t launch_decode_cluster4(DecodeArgs& a, const void* K, const void* V, cudaStream_t st);
cudaError_t launch_decode_cluster2(DecodeArgs& a, const void* K, const void* V, cudaStream_t st);

}  // namespace dash
