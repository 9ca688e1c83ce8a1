// Stage 2 backward, first pass (tensor cores, sm_100a): the log-sum-exp of every row's logits and delta = sum_j P_j dP_j
// (= <O, dO>), from S = Q K^T and dP = dO V^T alone.  Both are exact products of bf16 inputs accumulated in fp32, and the
// sums of exp(l) and exp(l) dP stay in fp32 registers: no O, no P V product, no rounding of P (delta feeds the gradient of
// the routing, which amplifies its error).
//
// Tile and walk as in the forward kernel (prefill_sm100.cu): 128 (token, head) rows, own chunks first, then the union of the
// rows' routed chunks, 64 keys per step.  Nothing flows back into the tensor cores, so the products run ahead of the sums: a
// ring of four K / V tiles and four S / dP slots (all 512 columns of tensor memory), a slot being free as soon as its
// values are in registers.  Three warpgroups take the steps in turn, each under a maximum of its own; a row's three parts meet
// at the end.
//
// Bound by the two score products: at N = 64 each MMA reads its 4 KiB slice of Q or dO again and holds the pipe 48 clocks,
// 768 per step.  8192 tokens, 32/8 heads, d 128: 397 us as a forward pass with two-term P, 385 us with one producer warp (900
// clocks a step, its pace), 410 with one issuer, 338 us; 2 x 1500 tokens, 8/2 heads, d 64, chunks of 32: 27 -> 18 us.
#include "bwd_sm100.cuh"

namespace dash {

namespace {

constexpr int NKV = BWD_NKV;
constexpr int THREADS = BWD_ROW_THREADS;
constexpr int RING = 4;                   // K / V tiles, step records, S / dP slots: index = step mod 4
constexpr uint32_t TMEM_COLS = 512, COL_DP = RING * NKV;      // S [0,256) dP [256,512)
constexpr float RESCALE_LOG2 = 8.f;       // a running maximum is moved only when it grew by more than this
enum Bar { QD_FULL = 0, META_READY, SD_FULL = 2, SD_FREE = 6, KV_FULL = 10, REC_FULL = 14, N_BARS = 18 };

template <int HD, int CPS, int MTQ>
struct Layout {
  struct Misc {
    unsigned long long bar[N_BARS];
    uint32_t tmem_base;
    int n_steps;
    int abort_flag;
    StepMeta<CPS, MTQ, RING, false> meta;
    float3 part[BWD_ROW_WG - 1][128];     // the other warpgroups' maxima and sums
  };
  static constexpr uint32_t Q_BYTES = 128 * HD * 2, KV_TILE_BYTES = NKV * HD * 2;
  static constexpr uint32_t OFF_Q = 0, OFF_DO = OFF_Q + Q_BYTES, OFF_K = OFF_DO + Q_BYTES, OFF_V = OFF_K + RING * KV_TILE_BYTES,
                            OFF_MISC = OFF_V + RING * KV_TILE_BYTES, SMEM = OFF_MISC + sizeof(Misc);
  static_assert(SMEM <= 232448, "one block per SM");
};

template <int HD, int CPS, int WT>
__global__ void __launch_bounds__(THREADS, 1)
attend_bwd_stats_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmDO,
                        const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, BwdArgs a) {
  constexpr int MTQ = 32 * (WT > 0 ? WT : 2);
  using LY = Layout<HD, CPS, MTQ>;
  using Misc = typename LY::Misc;
  constexpr uint32_t Q_BYTES = LY::Q_BYTES, KV_TILE_BYTES = LY::KV_TILE_BYTES, OFF_Q = LY::OFF_Q, OFF_DO = LY::OFF_DO;
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
    if (misc->abort_flag) report_error(a.sb, DASH_ERR_CUDA, 105);
    ptx::mbar_init(bar(QD_FULL), 1);
    ptx::mbar_init(bar(META_READY), 1);
    for (int s = 0; s < RING; ++s) {
      ptx::mbar_init(bar(SD_FULL + s), 1);
      ptx::mbar_init(bar(SD_FREE + s), 128);
      ptx::mbar_init(bar(KV_FULL + s), 1);
      ptx::mbar_init(bar(REC_FULL + s), 1);
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
  if (a.sb && *reinterpret_cast<volatile int*>(&a.sb->status) != 0) *abort_flag = 1;
  __syncthreads();

  if (warp >= BWD_W_TILES) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(bwd_regs_service(WT, CPS)));
    // everything of a step is free when its warpgroup has taken it (which both products precede)
    auto step_free = [&](int j) { return wait_all(bar(SD_FREE + j % RING), (uint32_t)(j / RING - 1) & 1u); };
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
      produce_steps<HD, CPS, WT, RING, RING, true, false>(
          a, &tmK, &tmV, grp, i0, lane, sbase + LY::OFF_K, sbase + LY::OFF_V, &misc->bar[KV_FULL], &misc->meta, a.inject != 0, step_free,
          [&](int n) {
            if (lane == 0) {
              misc->n_steps = n;
              ptx::mbar_arrive(bar(META_READY));
            }
          });
      if (lane == 0 && *abort_flag)
        for (int k = 0; k < 200000 && !ptx::mbar_try_wait(bar(QD_FULL), 0); ++k) {}
    } else if (warp == BWD_W_RECORDS) {
      produce_steps<HD, CPS, WT, RING, RING, false, false>(a, &tmK, &tmV, grp, i0, lane, 0u, 0u, &misc->bar[REC_FULL], &misc->meta,
                                                           false, step_free, [](int) {});
    } else {
      // two issuers of S = Q K^T and dP = dO V^T, of the even and the odd steps: between the products of a step and the next one's
      // lie some 250 clocks of barrier tests, which the other issuer's products fill
      const int parity = __shfl_sync(0xffffffffu, warp, 0) == BWD_W_SD ? 0 : 1;
      bool ok = wait_all(bar(QD_FULL), 0);
      int n_steps = 0x7fffffff;            // known from step 1 on; step 0 (the own chunk) always exists
      constexpr uint32_t IDESC_S = ptx::idesc_bf16_f32(128, NKV, false, false);
      const uint64_t qd = ptx::smem_desc_sw128(sbase + OFF_Q, 16, 1024), gd = ptx::smem_desc_sw128(sbase + OFF_DO, 16, 1024);
      const uint64_t kd0 = ptx::smem_desc_sw128(sbase + LY::OFF_K, 16, 1024), vd0 = ptx::smem_desc_sw128(sbase + LY::OFF_V, 16, 1024);
      const uint32_t d0 = __shfl_sync(0xffffffffu, tmem, 0);
      RingPos<RING> p;
      if (parity) p.step();
      for (int j = parity; j < n_steps && ok; j += 2, p.step(), p.step()) {
        if (j == 1 || j == 2) {
          ok = wait_all(bar(META_READY), 0);
          if (!ok) break;
          n_steps = __shfl_sync(0xffffffffu, misc->n_steps, 0);
          if (j >= n_steps) break;
        }
        // (the tiles' stage was refilled only after the threads had taken step j - 4, so the slot is free as well)
        ok = wait_all(bar(KV_FULL + p.at), p.phase);
        if (!ok) break;
        ptx::tc_fence_after();
        const uint64_t tile = (uint64_t)((p.at * KV_TILE_BYTES) >> 4);
        if (ptx::elect_one()) {
#pragma unroll
          for (int k = 0; k < HD / 16; ++k) {
            const uint64_t off_a = (uint64_t)(((k >> 2) * (Q_BYTES / 2) + (k & 3) * 32) >> 4);
            const uint64_t off_b = tile + (uint64_t)(((k >> 2) * (KV_TILE_BYTES / 2) + (k & 3) * 32) >> 4);
            ptx::mma_bf16_ss(d0 + p.at * NKV, qd + off_a, kd0 + off_b, IDESC_S, k > 0 ? 1u : 0u);
          }
#pragma unroll
          for (int k = 0; k < HD / 16; ++k) {
            const uint64_t off_a = (uint64_t)(((k >> 2) * (Q_BYTES / 2) + (k & 3) * 32) >> 4);
            const uint64_t off_b = tile + (uint64_t)(((k >> 2) * (KV_TILE_BYTES / 2) + (k & 3) * 32) >> 4);
            ptx::mma_bf16_ss(d0 + COL_DP + p.at * NKV, gd + off_a, vd0 + off_b, IDESC_S, k > 0 ? 1u : 0u);
          }
          ptx::mma_commit(bar(SD_FULL + p.at));
        }
        __syncwarp();
      }
    }
    __syncwarp();
  } else {
    // thread = tile row; warpgroup wg takes the steps wg, wg + 3, ...
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(bwd_regs_row(WT, CPS)));
    constexpr int W = NKV / CPS;                              // columns of a chunk slot
    const int wg = warp >> 2;
    const int m = (warp & 3) * 32 + lane;
    const int t = m / g_q, i_row = i0 + t;
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const float c1 = dm.sm_scale * LOG2E;
    float m_used = -INFINITY, l = 0.f, acc = 0.f;             // over this warpgroup's steps: maximum in use, sums of p and of p dP
    bool ok = true;
    int n_steps = 1;                                          // step 0 always exists; the others are known with the walk
    if (wg > 0) {
      ok = wait_all(bar(META_READY), 0);
      n_steps = ok ? misc->n_steps : 0;
    }
    for (int j = wg; j < n_steps && ok; j += BWD_ROW_WG) {
      const int st = j % RING;
      const uint32_t ph = (uint32_t)(j / RING) & 1u;
      ok = wait_all(bar(REC_FULL + st), ph);                  // the step's record is visible
      if (!ok) break;
      float b2[CPS];                                          // bias in the log2 domain (-inf: the row did not route the chunk)
      int n_vis[CPS];                                         // causal: column c of the slot visible iff c < n_vis
      bool any = false;
#pragma unroll
      for (int s = 0; s < CPS; ++s) {
        b2[s] = misc->meta.bias[st][s][t] * LOG2E;
        n_vis[s] = i_row - misc->meta.kvbase[st][s] + 1;
        any = any || b2[s] > -INFINITY;
      }
      ok = wait_all(bar(SD_FULL + st), ph);
      if (!ok) break;
      if (!__any_sync(0xffffffffu, any)) {                    // none of the warp's rows routed the step's chunks
        ptx::mbar_arrive(bar(SD_FREE + st));
      } else {
        ptx::tc_fence_after();
        uint32_t s0[32], s1[32], gv[32];
        DASH_TMEM_LD32(s0, lane_addr + st * NKV);
        DASH_TMEM_LD32(s1, lane_addr + st * NKV + 32);
        DASH_TMEM_WAIT_LD32(s0);
        DASH_TMEM_WAIT_LD32(s1);
        DASH_TMEM_LD32(gv, lane_addr + COL_DP + st * NKV);
        auto score = [&](int c) -> uint32_t& { return c < 32 ? s0[c & 31] : s1[c & 31]; };
        float mloc = -INFINITY;
#pragma unroll
        for (int s = 0; s < CPS; ++s) {
          if (b2[s] > -INFINITY) {
            if (n_vis[s] < W) {                               // only inside an own chunk
#pragma unroll
              for (int c = 0; c < W; ++c)
                if (c >= n_vis[s]) score(s * W + c) = 0xff800000u;
            }
            float ch[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) ch[c] = __uint_as_float(score(s * W + c));
#pragma unroll
            for (int c = 4; c < W; c += 4)
#pragma unroll
              for (int u = 0; u < 4; ++u) ch[u] = fmaxf(ch[u], __uint_as_float(score(s * W + c + u)));
            mloc = fmaxf(mloc, fmaf(fmaxf(fmaxf(ch[0], ch[1]), fmaxf(ch[2], ch[3])), c1, b2[s]));
          }
        }
        if (mloc > -INFINITY && (mloc > m_used + RESCALE_LOG2 || m_used == -INFINITY)) {
          const float corr = exp2f(m_used - mloc);            // 0 when nothing was accumulated yet
          l *= corr;
          acc *= corr;
          m_used = mloc;
        }
        const float2 c1v = make_float2(c1, c1);
        float2 ls[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}, as[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        // 32 columns: p = 2^(score - maximum), sums of p and p dP
        auto half = [&](int c0) {
          if (mloc > -INFINITY) {
#pragma unroll
            for (int c = 0; c < 32; c += 2) {
              const float o = b2[(c0 + c) / W] - m_used;
              const float2 x = __ffma2_rn(make_float2(__uint_as_float(score(c0 + c)), __uint_as_float(score(c0 + c + 1))), c1v, make_float2(o, o));
              const float2 p = make_float2(exp2f(x.x), exp2f(x.y));
              ls[(c >> 1) & 1] = __fadd2_rn(ls[(c >> 1) & 1], p);
              as[(c >> 1) & 1] = __ffma2_rn(p, make_float2(__uint_as_float(gv[c]), __uint_as_float(gv[c + 1])), as[(c >> 1) & 1]);
            }
          }
        };
        DASH_TMEM_WAIT_LD32(gv);
        half(0);
        DASH_TMEM_LD32(gv, lane_addr + COL_DP + st * NKV + 32);
        DASH_TMEM_WAIT_LD32(gv);
        ptx::tc_fence_before();
        ptx::mbar_arrive(bar(SD_FREE + st));
        half(32);
        const float2 lt = __fadd2_rn(ls[0], ls[1]), at = __fadd2_rn(as[0], as[1]);
        l += lt.x + lt.y;
        acc += at.x + at.y;
      }
      if (j == 0) {
        ok = wait_all(bar(META_READY), 0);
        n_steps = ok ? misc->n_steps : 0;
      }
    }
    if (wg > 0) misc->part[wg - 1][m] = make_float3(m_used, l, acc);
    asm volatile("bar.sync 1, %0;" ::"n"(BWD_ROW_WG * 128) : "memory");
    if (wg == 0 && ok && i_row < dm.seq_q) {
      const float3 o1 = misc->part[0][m], o2 = misc->part[1][m];
      const float mx = fmaxf(m_used, fmaxf(o1.x, o2.x));      // (a row sees at least its own key)
      const float w0 = exp2f(m_used - mx), w1 = exp2f(o1.x - mx), w2 = exp2f(o2.x - mx);
      const float lsum = fmaf(l, w0, fmaf(o1.y, w1, o2.y * w2)), dsum = fmaf(acc, w0, fmaf(o1.z, w1, o2.z * w2));
      *a.stats.at(b, r, i_row, m % g_q) = make_float2(mx + log2f(lsum), dsum / lsum);
    }
    ptx::tc_fence_before();
  }

  __syncthreads();
  if (misc->abort_flag) {                  // the kernels behind this one carry it on to every gradient of these rows
    for (int m = tid; m < 128; m += THREADS)
      if (i0 + m / g_q < dm.seq_q) *a.stats.at(b, r, i0 + m / g_q, m % g_q) = make_float2(gave_up(), gave_up());
  }
  if (warp == BWD_W_SD) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, TMEM_COLS);
  }
  if (tid == 0 && misc->abort_flag) report_error(a.sb, DASH_ERR_TIMEOUT, 106);
}

template <int HD, int CPS, int WT>
cudaError_t launch_one(const BwdArgs& a, const BwdMaps& m, cudaStream_t st) {
  auto kern = attend_bwd_stats_kernel<HD, CPS, WT>;
  constexpr uint32_t smem = Layout<HD, CPS, 32 * (WT > 0 ? WT : 2)>::SMEM;
  static std::atomic<unsigned long long> configured{0};
  if (cudaError_t e = allow_dynamic_smem(kern, smem, configured); e != cudaSuccess) return e;
  cudaError_t e = launch_chained(kern, dim3((unsigned)((long long)a.n_tiles * a.dm.batch * a.dm.h_kv)), dim3(THREADS), smem, st,
                                 m.q, m.g, m.kc, m.vc, a);
  count_launch();
  return e;
}

template <int HD, int CPS>
cudaError_t launch_cps(const BwdArgs& a, const BwdMaps& m, cudaStream_t st) {
  if (a.dm.g_q == 1) return launch_one<HD, CPS, 4>(a, m, st);
  if constexpr (CPS > 1) {
    if (a.TQ > a.dm.B) return launch_one<HD, CPS, 2>(a, m, st);
  }
  return launch_one<HD, CPS, 0>(a, m, st);
}

template <int HD>
cudaError_t launch_hd(const BwdArgs& a, const BwdMaps& m, cudaStream_t st) {
  if (a.dm.B >= NKV) return launch_cps<HD, 1>(a, m, st);
  return a.dm.B == 32 ? launch_cps<HD, 2>(a, m, st) : launch_cps<HD, 4>(a, m, st);
}

}  // namespace

cudaError_t launch_attend_bwd_stats(const BwdArgs& a, const BwdMaps& m, cudaStream_t st) {
  return a.dm.d == 128 ? launch_hd<128>(a, m, st) : launch_hd<64>(a, m, st);
}

}  // namespace dash
