// Stage 2, prefill, tensor-core path for sm_100a (Eq. 7 in the form of Proposition 1; Algorithm 3).
//
// Tile: one (batch, KV head) and TQ = 128/g_q consecutive query tokens; the rows of the MMA tile are (token,
// head-of-group) pairs, token-major.  Tiles start at multiples of TQ.  Where a chunk holds at least TQ tokens the tile's
// rows share their own chunk; where chunks are shorter (WIDE) the tile spans several, and every row has its own.  The own
// chunks go first (their tiles can be fetched before the mask has been read; each row sees its own one only, causally),
// then the tile walks the UNION of its rows' routed chunks in ascending order, 64 KV tokens per step.  A row that did
// not route a chunk gets bias -inf for that step (probability exactly 0), so every row still attends to its own
// selection only.
//
// Warp roles (256 threads = two warpgroups, two blocks per SM so one block's softmax overlaps the other's MMAs; after
// set-up the second warpgroup hands most of its registers to the first with setmaxnreg):
//   warps 0-3  softmax: S (TMEM) -> registers, logit = S/sqrt(d) + bias, causal mask inside the own chunk,
//              online softmax with a lazily moved row maximum, P (bf16) -> TMEM over the S columns, rescale of
//              the O accumulator in TMEM when the maximum moved, final O / l -> global.
//   warp 4     K producer: TMA loads of Q and of the K tiles (128-byte swizzle, no multicast); OR of the tile's
//              mask words = union list.
//   warp 6     V producer: walks the same union list; TMA loads of the V tiles and the per-token bias of each
//              step (a row's list entry for a chunk = its routed bits below the chunk + the totals of the earlier mask
//              words: read by direct index, a whole step's loads issued together before the wait for the stage).
//   warp 5     MMA issuer: S_{j+1} = Q K_{j+1}^T (M128 N64 K128) into one of two TMEM buffers, then O += P_j V_j
//              (M128 N128 K64, P from TMEM); one tcgen05.commit per product, to the mbarrier that the softmax
//              warps and the producer of the stage both listen to; owns the TMEM allocation.
//   warp 7     idle (it completes the second warpgroup: registers are re-divided per whole warpgroup).
// Every wait is bounded; a wait that runs out raises DASH_ERR_TIMEOUT in the status word and every role
// leaves its loop, frees TMEM and returns.
#include <cuda.h>

#include "common.cuh"
#include "sm100_ptx.cuh"
#include "tensor_map.cuh"
#include "tile_walk.cuh"

namespace dash {

namespace {

constexpr int NKV = 64;           // KV tokens per step
constexpr int KST = 2, VST = 2;   // ring depths: stage = step parity, like the S/P buffers, so that the two
                                  // MMA completion barriers of a step also release its K and V stages
constexpr int PF_THREADS = 256;   // 4 softmax warps, K producer, MMA issuer, V/bias producer and an idle warp: two whole
                                  // warpgroups, because a warpgroup changes its register budget only when all four of
                                  // its warps ask (a block of seven warps waits for the eighth for ever)
// Registers per thread after the re-division (two blocks per SM start with 128 each): what the
// softmax warpgroup takes is given up by the other one; the block's own pool is all that it can draw from.
// (A producer lane of a wide tile keeps every token's own chunk, and looks after four tokens where the tile has 128.)
__host__ __device__ constexpr int regs_service(int wt, int cps) { return wt > 2 ? (cps > 2 ? 96 : 88) : wt > 0 || cps > 2 ? 72 : 56; }
__host__ __device__ constexpr int regs_softmax(int wt, int cps) { return 256 - regs_service(wt, cps); }
static_assert(PF_THREADS == 256, "two warpgroups of equal size: one can take exactly what the other released");
constexpr uint32_t TMEM_COLS = 256;  // S0 [0,64), S1 [64,128), O [128,256)
constexpr float RESCALE_LOG2 = 8.f;  // the running maximum is moved only when it grew by more than this

// S_FULL[j&1]: QK of step j complete (S readable; K stage j&1 reusable).  PV_DONE[j&1]: PV of step j complete (O stable;
// S/P buffer and V stage j&1 reusable).  Every tcgen05.commit and every barrier test costs the issuing thread as
// much as an MMA, so each product signals exactly one barrier and the producers listen to the same ones.
enum Bar { Q_FULL = 0, META, S_FULL = 2, PV_DONE = 4, P_FULL = 6, V_FULL = 8, K_FULL = 10, N_BARS = 12 };
static_assert(KST == 2 && VST == 2, "stage = step parity");
// CPS = chunks per 64-token step: 1 for chunks of 64 or 128 tokens, 2 / 4 for chunks of 32 / 16 (a step then
// packs that many chunks of the union list, each with its own per-token bias).
// MTQ = most tokens a tile can hold.
template <int CPS, int MTQ>
struct MiscT {
  unsigned long long bar[N_BARS];
  uint32_t tmem_base;
  int n_steps;
  int abort_flag;
  int kvbase[VST][CPS];
  float bias[VST][CPS][MTQ];
};
// Shared-memory layout for head_dim HD (64 or 128): tiles are K-major regions of 64 elements (128 bytes, the
// swizzle span) per row, one region per 64 of head_dim.
template <int HD, int CPS, int MTQ>
struct PfLayout {
  static constexpr uint32_t Q_BYTES = 128 * HD * 2;           // HD = 128: 32 KiB, two 128x64 regions
  static constexpr uint32_t KV_TILE_BYTES = NKV * HD * 2;     // HD = 128: 16 KiB, two 64x64 regions
  static constexpr uint32_t OFF_Q = 0;
  static constexpr uint32_t OFF_K = OFF_Q + Q_BYTES;
  static constexpr uint32_t OFF_V = OFF_K + KST * KV_TILE_BYTES;
  static constexpr uint32_t OFF_MISC = OFF_V + VST * KV_TILE_BYTES;
  static constexpr uint32_t SMEM = OFF_MISC + sizeof(MiscT<CPS, MTQ>);
  static_assert(SMEM <= 115712, "two blocks per SM need <= 113 KiB each");
};


// max of three in one instruction
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

struct PrefillArgs {
  Dims dm;
  int TQ;            // tokens per tile
  int n_tiles;       // tiles per (batch, KV head)
  int early_loads;   // 1: Q, K, V are not written by the kernel before this one on the stream (their first loads may precede chain_wait)
  int resident;      // blocks that the device holds at once
  int inject;        // test hook: 1 = the K producer never loads the own chunk's keys (the waits for them run out)
  long long wait_limit;   // cycles a bounded wait may spin
  const uint32_t* mask;
  const float* blk_bias;
  __nv_bfloat16* O;
  StatusBlock* sb;
};

// WT > 0: a wide tile, which may span several chunks (chunks shorter than 128 / g_q tokens, or g_q = 1), of at most
// 32 * WT tokens; tiles inside one chunk (WT = 0, at most 64 tokens) compile without the per-row own chunks.
// P2: P enters the P V product as two bf16 terms (P = hi + lo, the remainder in the second half of the step's S columns),
// so O is accurate to fp32 class instead of bf16 class.  Taken for g_q = 1.
template <int HD, int CPS, int WT, bool P2>
__global__ void __launch_bounds__(PF_THREADS, 2)
attend_prefill_sm100_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                            const __grid_constant__ CUtensorMap tmV, PrefillArgs a) {
  constexpr bool WIDE = WT > 0;
  constexpr int TPL = WIDE ? WT : 2, MTQ = 32 * TPL;   // tokens a producer lane looks after: lane, lane + 32, ...
  constexpr int W = NKV / CPS;                         // KV tokens of one chunk slot of a step
  using LY = PfLayout<HD, CPS, MTQ>;
  using Misc = MiscT<CPS, MTQ>;
  constexpr uint32_t Q_BYTES = LY::Q_BYTES, KV_TILE_BYTES = LY::KV_TILE_BYTES, OFF_Q = LY::OFF_Q, OFF_K = LY::OFF_K,
                     OFF_V = LY::OFF_V, OFF_MISC = LY::OFF_MISC;
  extern __shared__ __align__(1024) uint8_t smem[];
  Misc* misc = reinterpret_cast<Misc*>(smem + OFF_MISC);
  const Dims& dm = a.dm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t sbase = ptx::smem_u32(smem);
  auto bar = [&](int i) { return ptx::smem_u32(&misc->bar[i]); };
  volatile int* abort_flag = &misc->abort_flag;
  const long long wait_limit = a.wait_limit;
  auto wait_on = [&](uint32_t barrier, uint32_t parity) { return ptx::mbar_wait(barrier, parity, abort_flag, wait_limit); };
  auto wait_all = [&](uint32_t barrier, uint32_t parity) { return ptx::mbar_wait_warp(barrier, parity, abort_flag, wait_limit); };

  const int groups = dm.batch * dm.h_kv;
  const int tile = a.n_tiles - 1 - (int)(blockIdx.x / groups);  // late (long) tiles first
  const int grp = (int)(blockIdx.x % groups);
  const int b = grp / dm.h_kv, r = grp % dm.h_kv;
  const int TQ = a.TQ, g_q = dm.g_q;
  const int i0 = tile * TQ;
  const int c_own = i0 >> dm.log_b;                        // own chunk of the tile's first token (WIDE: of that one only)
  const int sub_per_blk = dm.B / NKV;                 // 64-token steps per chunk (1 or 2)
  const int own_steps = WIDE ? (TQ + NKV - 1) / NKV   // steps over the tile's own tokens
                             : (i0 % dm.B) / NKV + 1; // steps of the own chunk the tile can see

  if (tid == 0) {
    if ((sbase & 1023u) != 0u) {
      report_error(a.sb, DASH_ERR_CUDA, 100);
      misc->abort_flag = 1;
    } else {
      misc->abort_flag = 0;
    }
    ptx::mbar_init(bar(Q_FULL), 1);
    ptx::mbar_init(bar(META), 1);
    for (int s = 0; s < 2; ++s) {
      ptx::mbar_init(bar(S_FULL + s), 1);
      ptx::mbar_init(bar(PV_DONE + s), 1);
      ptx::mbar_init(bar(K_FULL + s), 1);
      ptx::mbar_init(bar(V_FULL + s), 1);
    }
    // two P_FULL barriers (step parity): the softmax warps may finish step j+1 before the MMA thread has
    // looked at step j, and a single barrier's phase bit cannot tell j from j+2
    ptx::mbar_init(bar(P_FULL), 128);
    ptx::mbar_init(bar(P_FULL + 1), 128);
    ptx::fence_barrier_init();
  }
  if (warp == 5) {
    ptx::tmem_alloc(ptx::smem_u32(&misc->tmem_base), TMEM_COLS);
    ptx::tmem_relinquish();
    ptx::tc_fence_before();
  }
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = misc->tmem_base;
  // A step's K or V tile for chunks smaller than the step: CPS boxes of NKV / CPS tokens, one per packed chunk.
  [[maybe_unused]] auto load_packed = [&](const CUtensorMap* tm, uint32_t dst, uint32_t barrier, const int* kvs) {
    ptx::mbar_arrive_expect_tx(barrier, KV_TILE_BYTES);
#pragma unroll
    for (int s = 0; s < CPS; ++s) {
      const uint32_t d = dst + s * (NKV / CPS) * 128;
      ptx::tma_load_4d(d, tm, barrier, 0, r, kvs[s], b);
      if constexpr (HD == 128) ptx::tma_load_4d(d + KV_TILE_BYTES / 2, tm, barrier, 64, r, kvs[s], b);
    }
  };
  // Q and the own chunk's K / V tiles: they need nothing from the routing kernels (and go first anyway).
  auto own_loads = [&](bool do_k, bool do_v) {
    if (lane == 0 && do_k) {
      ptx::prefetch_tensormap(&tmQ);
      ptx::prefetch_tensormap(&tmK);
      ptx::prefetch_tensormap(&tmV);
      ptx::mbar_arrive_expect_tx(bar(Q_FULL), Q_BYTES);
      ptx::tma_load_4d(sbase + OFF_Q, &tmQ, bar(Q_FULL), 0, r * g_q, i0, b);
      if constexpr (HD == 128) ptx::tma_load_4d(sbase + OFF_Q + Q_BYTES / 2, &tmQ, bar(Q_FULL), 64, r * g_q, i0, b);
    }
    // The own chunk goes first: its tiles need nothing from the mask, so they are in flight (and the first
    // S = Q K^T can run) while the union of the routed chunks is still being formed.  Stages 0/1 are free.
    for (int sub = 0; sub < own_steps; ++sub) {
      // narrow tile: the own chunk fills the first slot, the other slots repeat it; wide tile: its own chunks in order
      // (slots behind its last token repeat the first chunk).  bias 0 where the slot is the token's own chunk, -inf elsewhere
      int kvs[CPS];
      const int kv0 = WIDE ? i0 + sub * NKV : c_own * dm.B + sub * NKV;
#pragma unroll
      for (int s = 0; s < CPS; ++s) kvs[s] = WIDE && kv0 + s * W < i0 + TQ ? kv0 + s * W : kv0;
      if (do_k) {
        if (lane == 0 && !a.inject) load_packed(&tmK, sbase + OFF_K + sub * KV_TILE_BYTES, bar(K_FULL + sub), kvs);
      } else {
        for (int t = lane; t < TQ; t += 32)
#pragma unroll
          for (int s = 0; s < CPS; ++s)
            misc->bias[sub][s][t] = (WIDE ? (kv0 + s * W) >> dm.log_b == (i0 + t) >> dm.log_b : s == 0) ? 0.f : -INFINITY;
#pragma unroll
        for (int s = 0; s < CPS; ++s)
          if (lane == s) misc->kvbase[sub][s] = kvs[s];
        __syncwarp();
        if (lane == 0) load_packed(&tmV, sbase + OFF_V + sub * KV_TILE_BYTES, bar(V_FULL + sub), kvs);
      }
    }
  };
  // Q, K and V are inputs of the whole chain, not outputs of the kernel before this one: when the caller vouches for
  // that, their first tiles are under way while that kernel still drains
  if (a.early_loads && (warp == 4 || warp == 6)) own_loads(warp == 4, warp == 6);
  // barriers and tensor memory are set up; from here on the kernel reads what the routing kernels wrote
  chain_wait();
  // The next kernel's blocks: at once where this grid takes several waves (they come with its last one), else only when this
  // block is done, for they would all settle on the SMs that have none of the few blocks (500 tokens: 24.7 -> 23.6 us a forward).
  const bool release_late = (int)gridDim.x <= a.resident;
  if (!release_late) chain_release();
  // a workspace whose status word already holds an error makes every role leave at its first wait: after one
  // block's wait has run out, the rest of the grid retires in microseconds instead of a wait limit each
  if (a.sb && *reinterpret_cast<volatile int*>(&a.sb->status) != 0) *abort_flag = 1;
  __syncthreads();

  if (warp >= 4) {
  // the register file of the block is re-divided between its two warpgroups: this one gives up what the softmax
  // warpgroup takes (each side opens with its own instruction, so the allocator knows the budget of each)
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(regs_service(WT, CPS)));
  if (warp == 4 || warp == 6) {
    // =========================== producers ===========================
    // Two warps walk the same union list: warp 4 feeds the K ring (and loads Q), warp 6 feeds the V ring and
    // the per-token bias of each step.  Split like this, a full V ring never holds back the next K tile.
    const bool do_k = (warp == 4), do_v = (warp == 6);
    if (!a.early_loads) own_loads(do_k, do_v);
    TileWalk<CPS, WIDE, TPL> walk(dm, a.mask, ((long long)b * dm.h_kv + r) * dm.seq_q, i0, TQ, lane);
    const int total = walk.count();
    const int n_steps = (CPS > 1 ? (total + CPS - 1) / CPS : total * sub_per_blk) + own_steps;
    if (lane == 0 && do_k) {
      misc->n_steps = n_steps;
      ptx::mbar_arrive(bar(META));
    }
    // the compact bias lists of this lane's tokens
    const float* list[TPL];
#pragma unroll
    for (int q = 0; q < TPL; ++q)
      list[q] = a.blk_bias + ((long long)b * dm.h_kv + r) * dm.list_rows + list_row_offset(dm, min(i0 + lane + 32 * q, dm.seq_q - 1));
    walk.start();
    bool ok = true;
    // last step loaded into each stage (-1: none): what a block that gives up has to let land before it retires
    int last_j[2] = {-1, -1};
    for (int sub = 0; sub < own_steps; ++sub) last_j[sub] = (do_k && a.inject) ? -1 : sub;
    for (int j = own_steps; j < n_steps && ok;) {      // (the own chunks' steps are already under way)
      // a step takes the next CPS chunks of the union (CPS > 1: chunks of 32 / 16 tokens packed into the 64-token step);
      // the bias loads of a whole step are issued together, before the wait for the stage
      int cs[CPS], pos[CPS][TPL];
      float bvs[CPS][TPL];
      walk.next(cs, pos);
      if (do_v) {
#pragma unroll
        for (int s = 0; s < CPS; ++s)
#pragma unroll
          for (int q = 0; q < TPL; ++q) bvs[s][q] = pos[s][q] >= 0 ? __ldg(list[q] + pos[s][q]) : -INFINITY;
      }
      // chunks of 128 tokens take two 64-token steps with the same bias
      for (int sub = 0; sub < (CPS > 1 ? 1 : sub_per_blk) && ok; ++sub, ++j) {
        int kvs[CPS];
#pragma unroll
        for (int s = 0; s < CPS; ++s) kvs[s] = cs[s] * dm.B + sub * NKV;
        const int st = j & 1, prev_ph = ((j >> 1) - 1) & 1;   // stage, and the phase of step j-2 on the completion barriers
        if (do_k) {
          if (j >= 2) ok = wait_all(bar(S_FULL + st), prev_ph);    // QK of step j-2 has read the stage
          if (!ok) break;
          if (lane == 0) load_packed(&tmK, sbase + OFF_K + st * KV_TILE_BYTES, bar(K_FULL + st), kvs);
        } else {
          const bool free = j < 2 || wait_on(bar(PV_DONE + st), prev_ph);    // PV of step j-2 has read the stage
#pragma unroll
          for (int s = 0; s < CPS; ++s) {
#pragma unroll
            for (int q = 0; q < TPL; ++q) {
              const int t = lane + 32 * q;
              if (t < TQ) misc->bias[st][s][t] = bvs[s][q];
            }
            if (lane == s) misc->kvbase[st][s] = kvs[s];
          }
          ok = __all_sync(0xffffffffu, free);      // (the record is written, too; nobody reads it if the warp gives up)
          if (!ok) break;
          if (lane == 0) load_packed(&tmV, sbase + OFF_V + st * KV_TILE_BYTES, bar(V_FULL + st), kvs);
        }
        last_j[st] = j;
      }
    }
    if (!ok && lane == 0) {
      // a wait ran out: let the copies already issued land (bounded) before the block retires
      for (int s = 0; s < 2; ++s) {
        if (last_j[s] < 0) continue;
        const uint32_t full = bar((do_k ? K_FULL : V_FULL) + s), parity = (uint32_t)(last_j[s] >> 1) & 1u;
        for (int k = 0; k < 200000 && !ptx::mbar_try_wait(full, parity); ++k) {}
      }
      if (do_k)
        for (int k = 0; k < 200000 && !ptx::mbar_try_wait(bar(Q_FULL), 0); ++k) {}
    }
  } else if (warp == 5) {
    // =========================== MMA issuer ===========================
    // Per step: S_{j+1} = Q K_{j+1}^T (needs only its K tile), then O += P_j V_j.  V_FULL is not tested here: the
    // softmax threads wait for it (the step's bias arrives with it) before they arrive on P_FULL.
    if (lane == 0) {
      bool ok = wait_on(bar(Q_FULL), 0);
      constexpr uint32_t IDESC_QK = ptx::idesc_bf16_f32(128, NKV, false, false);
      constexpr uint32_t IDESC_PV = ptx::idesc_bf16_f32(128, HD, false, true);
      // Descriptors differ only in the 14-bit start-address field (16-byte units, no carry into the next
      // field): build them once, then a single add per MMA keeps the issuing thread's instruction stream short.
      const uint64_t qd0 = ptx::smem_desc_sw128(sbase + OFF_Q, 16, 1024);
      const uint64_t kd0 = ptx::smem_desc_sw128(sbase + OFF_K, 16, 1024);
      const uint64_t vd0 = ptx::smem_desc_sw128(sbase + OFF_V, KV_TILE_BYTES / 2, 1024);
      auto issue_qk = [&](int j) -> bool {
        const int buf = j & 1;
        if (!wait_on(bar(K_FULL + buf), (j >> 1) & 1)) return false;
        // the S/P buffer is recycled in MMA issue order (PV of step j-2 precedes this QK)
        ptx::tc_fence_after();
        const uint64_t kd = kd0 + (uint64_t)((buf * KV_TILE_BYTES) >> 4);
        const uint32_t d_tmem = tmem + buf * NKV;
#pragma unroll
        for (int k = 0; k < HD / 16; ++k) {
          // 16 bf16 = 32 bytes inside the 128-byte swizzle row; the second 64 columns live in the next region
          const uint64_t ad = qd0 + (uint64_t)(((k >> 2) * (Q_BYTES / 2) + (k & 3) * 32) >> 4);
          const uint64_t bd = kd + (uint64_t)(((k >> 2) * (KV_TILE_BYTES / 2) + (k & 3) * 32) >> 4);
          ptx::mma_bf16_ss(d_tmem, ad, bd, IDESC_QK, k > 0 ? 1u : 0u);
        }
        ptx::mma_commit(bar(S_FULL + buf));
        return true;
      };
      if (ok) ok = issue_qk(0);          // the own chunk: there is always a step 0, whatever the union holds
      ok = ok && wait_on(bar(META), 0);
      const int n_steps = ok ? misc->n_steps : 0;
      for (int j = 0; j < n_steps && ok; ++j) {
        if (j + 1 < n_steps) ok = issue_qk(j + 1);
        if (!ok) break;
        const int buf = j & 1;
        ok = wait_on(bar(P_FULL + buf), (j >> 1) & 1);
        if (!ok) break;
        ptx::tc_fence_after();
        // V is [kv token][d]: MN-major B operand; 64-wide d blocks are KV_TILE_BYTES/2 apart; 16 tokens = 2048 bytes
        const uint64_t vd = vd0 + (uint64_t)((buf * KV_TILE_BYTES) >> 4);
        const uint32_t p_tmem = tmem + buf * NKV;
#pragma unroll
        for (int k = 0; k < NKV / 16; ++k) {
          const uint64_t bd = vd + (uint64_t)((k * 16 * 128) >> 4);
          // A = P from tensor memory: 16 bf16 per K step = 8 packed columns
          ptx::mma_bf16_ts(tmem + 2 * NKV, p_tmem + k * 8, bd, IDESC_PV, (j > 0 || k > 0) ? 1u : 0u);
        }
        if constexpr (P2) {
#pragma unroll
          for (int k = 0; k < NKV / 16; ++k) {
            const uint64_t bd = vd + (uint64_t)((k * 16 * 128) >> 4);
            ptx::mma_bf16_ts(tmem + 2 * NKV, p_tmem + 32 + k * 8, bd, IDESC_PV, 1u);      // the remainders
          }
        }
        ptx::mma_commit(bar(PV_DONE + buf));
      }
    }
    __syncwarp();
  }
  } else {
    // =========================== softmax / epilogue ===========================
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(regs_softmax(WT, CPS)));
    const int m = tid;                       // tile row = TMEM lane
    const int t = m / g_q, hh = m % g_q;     // token in tile, head in group
    const int i_row = i0 + t;
    const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
    const float c1 = dm.sm_scale * 1.4426950408889634f;
    bool ok = true;
    int n_steps = 0x7fffffff;                // known from step 1 on; step 0 (the own chunk) always exists
    float m_used = -INFINITY, l = 0.f;

    for (int j = 0; ok; ++j) {
      if (j == 1) {
        ok = wait_all(bar(META), 0);
        if (!ok) break;
        n_steps = misc->n_steps;
      }
      if (j >= n_steps) break;
      const int buf = j & 1;
      // bias / kvbase of the step visible; the MMA thread relies on this wait for the V tile as well.  (A lane whose wait runs out
      // here or at the scores stays with its warp, on values of no meaning, until the warp votes before it hands P on.)
      bool here = wait_on(bar(V_FULL + buf), (j >> 1) & 1);
      float b2s[CPS];                                // per packed chunk: bias in the log2 domain (-inf: not routed)
#pragma unroll
      for (int s = 0; s < CPS; ++s) b2s[s] = misc->bias[buf][s][t] * 1.4426950408889634f;
      const int kv0 = misc->kvbase[buf][0];
      here = wait_on(bar(S_FULL + buf), (j >> 1) & 1) && here;
      ptx::tc_fence_after();
      uint32_t sreg[64];
      {
        uint32_t* lo = sreg;
        uint32_t* hi = sreg + 32;
        DASH_TMEM_LD32(lo, lane_addr + buf * NKV);
        DASH_TMEM_LD32(hi, lane_addr + buf * NKV + 32);
      }
      ptx::tmem_wait_ld();

      // logit (log2 domain) = s*c1 + b2; c1 > 0, so the row maximum can be taken on the raw scores
      const int n_vis = i_row - kv0 + 1;             // causal: KV token kv0 + c visible iff c < n_vis
      bool selected;
      float mloc;
      if constexpr (CPS > 1) {
        // packed chunks: each slot of W columns has its own bias; only a slot of an own chunk can be cut by the causal
        // mask (routed chunks lie wholly before the row): slot 0 of step 0, in a wide tile every slot of the first steps
        mloc = -INFINITY;
#pragma unroll
        for (int s = 0; s < CPS; ++s) {
          if (b2s[s] > -INFINITY) {
            const int vis = s == 0 ? n_vis : WIDE && j < own_steps ? i_row - misc->kvbase[buf][s] + 1 : W;
            if (vis < W) {
#pragma unroll
              for (int c = 0; c < W; ++c)
                if (c >= vis) sreg[s * W + c] = 0xff800000u;   // -inf
            }
            float ch[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) ch[c] = __uint_as_float(sreg[s * W + c]);
#pragma unroll
            for (int k = 4; k < W; k += 4)
#pragma unroll
              for (int c = 0; c < 4; ++c) ch[c] = fmaxf(ch[c], __uint_as_float(sreg[s * W + c + k]));
            mloc = fmaxf(mloc, fmaf(fmaxf(fmaxf(ch[0], ch[1]), fmaxf(ch[2], ch[3])), c1, b2s[s]));
          }
        }
        selected = mloc > -INFINITY;
      }
      const float b2 = b2s[0];
      float mr = -INFINITY;
      if constexpr (CPS == 1) selected = b2 > -INFINITY;
      if (CPS == 1 && selected) {
        if (n_vis < NKV) {                           // only inside the own chunk
#pragma unroll
          for (int c = 0; c < NKV; ++c)
            if (c >= n_vis) sreg[c] = 0xff800000u;   // -inf
        }
        // three-input maxima: 32 instructions for the 64 scores, in eight independent chains, then a tree
        float ch[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) ch[c] = __uint_as_float(sreg[c]);
#pragma unroll
        for (int k = 8; k + 16 <= NKV; k += 16)
#pragma unroll
          for (int c = 0; c < 8; ++c) ch[c] = max3(ch[c], __uint_as_float(sreg[c + k]), __uint_as_float(sreg[c + k + 8]));
#pragma unroll
        for (int c = 0; c < 8; ++c) ch[c] = fmaxf(ch[c], __uint_as_float(sreg[c + NKV - 8]));
        mr = fmaxf(max3(ch[0], ch[1], ch[2]), fmaxf(max3(ch[3], ch[4], ch[5]), fmaxf(ch[6], ch[7])));
      }
      if constexpr (CPS == 1) mloc = fmaf(mr, c1, b2);           // -inf when not selected
      float corr = 1.f;
      bool moved = false;
      if (mloc > m_used + RESCALE_LOG2 || (m_used == -INFINITY && mloc > -INFINITY)) {
        corr = exp2f(m_used - mloc);   // 0 when nothing was accumulated yet
        m_used = mloc;
        moved = true;
      }
      l *= corr;
      [[maybe_unused]] uint32_t packed[P2 ? 1 : 32];
      if constexpr (P2) {
        // P = hi + lo as two bf16 terms, 32 scores at a time, stored as they are formed (the scores are all in registers
        // already): hi into the first 32 columns of the step's S buffer, lo into the second 32
        float2 lsum[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        const float2 c1v = make_float2(c1, c1);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          uint32_t hi16[16], lo16[16];
          if (selected) {
#pragma unroll
            for (int c = 0; c < 32; c += 2) {
              const int cc = half * 32 + c;
              const float2 offv = make_float2(b2s[cc / W] - m_used, b2s[cc / W] - m_used);
              const float2 t = __ffma2_rn(make_float2(__uint_as_float(sreg[cc]), __uint_as_float(sreg[cc + 1])), c1v, offv);
              const float2 pp = make_float2(exp2f(t.x), exp2f(t.y));
              lsum[(c >> 1) & 1] = __fadd2_rn(lsum[(c >> 1) & 1], pp);
              __nv_bfloat162 h = __floats2bfloat162_rn(pp.x, pp.y);
              const float2 hf = __bfloat1622float2(h);
              __nv_bfloat162 lo = __floats2bfloat162_rn(pp.x - hf.x, pp.y - hf.y);
              hi16[c >> 1] = *reinterpret_cast<uint32_t*>(&h);
              lo16[c >> 1] = *reinterpret_cast<uint32_t*>(&lo);
            }
          } else {
#pragma unroll
            for (int c = 0; c < 16; ++c) hi16[c] = lo16[c] = 0u;
          }
          ptx::tmem_st_n<16>(lane_addr + buf * NKV + half * 16, hi16);
          ptx::tmem_st_n<16>(lane_addr + buf * NKV + 32 + half * 16, lo16);
        }
        const float2 ls = __fadd2_rn(lsum[0], lsum[1]);
        l += ls.x + ls.y;
      } else if (selected) {
        // scale-and-shift and the row sum on packed pairs (one instruction per two scores); a slot that is not
        // routed has offset -inf, so its probabilities come out as exactly 0
        const float2 c1v = make_float2(c1, c1);
        float2 offs[CPS];
#pragma unroll
        for (int s = 0; s < CPS; ++s) offs[s] = make_float2(b2s[s] - m_used, b2s[s] - m_used);
        float2 lsum[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int c = 0; c < NKV; c += 2) {
          const float2 offv = offs[c / W];
          const float2 t = __ffma2_rn(make_float2(__uint_as_float(sreg[c]), __uint_as_float(sreg[c + 1])), c1v, offv);
          const float2 pp = make_float2(exp2f(t.x), exp2f(t.y));
          lsum[(c >> 1) & 3] = __fadd2_rn(lsum[(c >> 1) & 3], pp);
          __nv_bfloat162 h = __floats2bfloat162_rn(pp.x, pp.y);
          packed[c >> 1] = *reinterpret_cast<uint32_t*>(&h);
        }
        const float2 ls = __fadd2_rn(__fadd2_rn(lsum[0], lsum[1]), __fadd2_rn(lsum[2], lsum[3]));
        l += ls.x + ls.y;
      } else {
#pragma unroll
        for (int c = 0; c < 32; ++c) packed[c] = 0u;
      }

      // O is stable once the previous step's PV has completed
      const bool fix = __any_sync(0xffffffffu, moved || !here);
      if (fix) {
        ok = __all_sync(0xffffffffu, here);
        if (!ok) break;
      }
      if (fix && j > 0) {
        ok = wait_all(bar(PV_DONE + (buf ^ 1)), ((j - 1) >> 1) & 1);
        if (!ok) break;
        ptx::tc_fence_after();
        // rescale this row of the accumulator: O *= 2^(m_old - m_new)
#pragma unroll 1
        for (int q = 0; q < HD / 32; ++q) {
          uint32_t o[32];
          DASH_TMEM_LD32(o, lane_addr + 2 * NKV + q * 32);
          ptx::tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * corr);
          DASH_TMEM_ST32(lane_addr + 2 * NKV + q * 32, o);
        }
      }
      // P row -> the first 32 columns of this step's S buffer (two bf16 per column)
      if constexpr (!P2) DASH_TMEM_ST32(lane_addr + buf * NKV, packed);
      ptx::tmem_wait_st();
      ptx::tc_fence_before();
      ptx::mbar_arrive(bar(P_FULL + (j & 1)));
    }

    // epilogue: O / l -> global (row m is 128 contiguous bf16 of token i_row, head r*g_q + hh)
    if (ok && n_steps > 0) ok = wait_all(bar(PV_DONE + ((n_steps - 1) & 1)), ((n_steps - 1) >> 1) & 1);
    if (ok && n_steps > 0) {
      ptx::tc_fence_after();
      const float inv = l > 0.f ? 1.f / l : 0.f;
      __nv_bfloat16* op = a.O + (long long)b * dm.os[0] + (long long)i_row * dm.os[1] + (long long)(r * g_q + hh) * dm.os[2];
      const bool row_out = i_row < dm.seq_q;
#pragma unroll 1
      for (int q = 0; q < HD / 32; ++q) {
        uint32_t o[32];
        DASH_TMEM_LD32(o, lane_addr + 2 * NKV + q * 32);
        ptx::tmem_wait_ld();
        if (row_out) {
#pragma unroll
          for (int c = 0; c < 32; c += 8) {
            uint4 v;
            __nv_bfloat162 h0 = __floats2bfloat162_rn(__uint_as_float(o[c]) * inv, __uint_as_float(o[c + 1]) * inv);
            __nv_bfloat162 h1 = __floats2bfloat162_rn(__uint_as_float(o[c + 2]) * inv, __uint_as_float(o[c + 3]) * inv);
            __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(o[c + 4]) * inv, __uint_as_float(o[c + 5]) * inv);
            __nv_bfloat162 h3 = __floats2bfloat162_rn(__uint_as_float(o[c + 6]) * inv, __uint_as_float(o[c + 7]) * inv);
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
  if (release_late) chain_release();
  if (warp == 5) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, TMEM_COLS);
  }
  if (tid == 0 && misc->abort_flag) report_error(a.sb, DASH_ERR_TIMEOUT, 101);
}

// ---------------------------------------------------------------- host side

// [batch, tokens, heads, 128] bf16 tensor with element strides s[3]; box = 64 x box_heads x box_tokens x 1.
bool make_map(CUtensorMap* out, const void* base, int hd, long long tokens, int heads, int batch, const long long* s,
              int box_heads, int box_tokens) {
  cuuint64_t dims[4] = {(cuuint64_t)hd, (cuuint64_t)heads, (cuuint64_t)tokens, (cuuint64_t)batch};
  // a size-1 dimension may come with stride 0; any positive multiple of 16 bytes is accepted there
  auto st = [](long long e) { return (cuuint64_t)((e > 0 ? e : 8) * 2); };
  cuuint64_t strides[3] = {st(s[2]), st(s[1]), st(s[0])};
  cuuint32_t box[4] = {64u, (cuuint32_t)box_heads, (cuuint32_t)box_tokens, 1u};
  return encode_bf16_sw128_4d(out, base, dims, strides, box);
}

}  // namespace

bool prefill_sm100_supported(const Dims& dm) {
  if (dm.decode || !dm.causal || dm.dtype != DASH_BF16 || (dm.d != 64 && dm.d != 128)) return false;
  if (dm.B != 16 && dm.B != 32 && dm.B != 64 && dm.B != 128) return false;
  if (dm.os[2] % 8 != 0 || dm.os[1] % 8 != 0) return false;
  if (broadcasts(dm.qs, dm.batch, dm.seq_q, dm.h_q) || broadcasts(dm.ks, dm.batch, dm.seq_kv, dm.h_kv) ||
      broadcasts(dm.vs, dm.batch, dm.seq_kv, dm.h_kv))
    return false;
  return tensor_map_encoder() != nullptr;
}

template <int HD, int CPS, int WT, bool P2>
static cudaError_t launch_one(const PrefillArgs& a, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                              cudaStream_t st) {
  auto kern = attend_prefill_sm100_kernel<HD, CPS, WT, P2>;
  constexpr uint32_t smem = PfLayout<HD, CPS, 32 * (WT > 0 ? WT : 2)>::SMEM;
  static std::atomic<unsigned long long> configured{0};
  if (cudaError_t e = allow_dynamic_smem(kern, smem, configured); e != cudaSuccess) return e;
  const unsigned blocks = (unsigned)((long long)a.n_tiles * a.dm.batch * a.dm.h_kv);
  cudaError_t e = launch_chained(kern, dim3(blocks), dim3(PF_THREADS), smem, st, tq, tk, tv, a);
  count_launch();
  return e;
}

// Tiles of 128 / g_q tokens: g_q = 1 takes the 128-token wide form with two-term probabilities (the precision it had on
// CUDA cores), chunks shorter than the tile the 64-token wide form.  A tile that keeps all 128 rows live over several
// chunks walks a larger union than one cut at the chunk's end, but there are fewer tiles and no dead rows: 8192 tokens,
// 32/8 heads, chunks of 16: 1.43 -> 0.58 ms; 3 x 1999 tokens, 12/12 heads, d 64, chunks of 32: 1.54 ms on CUDA cores
// (one warp per row) -> 0.07 ms.
template <int HD, int CPS>
static cudaError_t launch_cps(const PrefillArgs& a, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                              cudaStream_t st) {
  if (a.dm.g_q == 1) return launch_one<HD, CPS, 4, true>(a, tq, tk, tv, st);
  if constexpr (CPS > 1) {
    if (a.TQ > a.dm.B) return launch_one<HD, CPS, 2, false>(a, tq, tk, tv, st);
  }
  return launch_one<HD, CPS, 0, false>(a, tq, tk, tv, st);
}

template <int HD>
static cudaError_t launch_hd(const PrefillArgs& a, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                             cudaStream_t st) {
  if (a.dm.B >= NKV) return launch_cps<HD, 1>(a, tq, tk, tv, st);
  return a.dm.B == 32 ? launch_cps<HD, 2>(a, tq, tk, tv, st) : launch_cps<HD, 4>(a, tq, tk, tv, st);
}

cudaError_t launch_attend_prefill_sm100(const Dims& dm, const void* Q, const void* K, const void* V,
                                        const uint32_t* mask, const float* blk_bias, void* O, StatusBlock* sb,
                                        bool inputs_stable, cudaStream_t st) {
  PrefillArgs a;
  a.dm = dm;
  a.TQ = 128 / dm.g_q;
  a.n_tiles = (dm.seq_q + a.TQ - 1) / a.TQ;
  a.early_loads = inputs_stable ? 1 : 0;
  a.resident = 2 * current_sm_count();
  a.inject = test_hooks().skip_own_k_load;
  a.wait_limit = test_hooks().wait_limit_cycles;
  a.mask = mask;
  a.blk_bias = blk_bias;
  a.O = (__nv_bfloat16*)O;
  a.sb = sb;
  CUtensorMap tq, tk, tv;
  const int box_kv = dm.B < NKV ? dm.B : NKV;      // chunks below 64 tokens are fetched one box per chunk
  if (!make_map(&tq, Q, dm.d, dm.seq_q, dm.h_q, dm.batch, dm.qs, dm.g_q, a.TQ)) return cudaErrorInvalidValue;
  if (!make_map(&tk, K, dm.d, dm.seq_kv, dm.h_kv, dm.batch, dm.ks, 1, box_kv)) return cudaErrorInvalidValue;
  if (!make_map(&tv, V, dm.d, dm.seq_kv, dm.h_kv, dm.batch, dm.vs, 1, box_kv)) return cudaErrorInvalidValue;
  return dm.d == 128 ? launch_hd<128>(a, tq, tk, tv, st) : launch_hd<64>(a, tq, tk, tv, st);
}

}  // namespace dash
