// Backward of Stage 1 (routing) and Stage 0 (chunk summaries), prefill, on CUDA cores.
//
// Section 3.5 notes that the backward pass can reuse the forward pass's bit mask because the alpha-entmax Jacobian is
// sparse; the appendix ("The alpha-entmax mapping") states that the Jacobian has a closed form where the support is
// fixed.  From Eq. 2, p_c = [(alpha-1) z_c - tau]_+^(1/(alpha-1)) with sum_c p_c = 1: on the support
// dp_c = s_c (dz_c - dtau/(alpha-1)) with s_c = p_c^(2-alpha) = margin_c^(1/(alpha-1) - 1), and sum dp = 0 fixes
// dtau, so dz = s * (dp - <s, dp> / sum(s)) and nothing outside the support receives or passes on a gradient.
//
// route_bwd_kernel: one warp per (batch, KV head, query row).  Input: the row's routed chunk list (chunk ids), the
// thresholds tau of the group's heads, and dbias (gradient w.r.t. the log-prior bias of every routed chunk, from the
// Stage-2 backward).  Chain rule of Section 3.2 / Proposition 1:
//   bias_c = (log w_c - mean_S log w)/sigma  =>  dlogw_c = (dbias_c - mean_S dbias)/sigma,  dw_c = dlogw_c / w_c
//   w_c = mean_h p_hc                        =>  dp_hc = dw_c / g_q
//   p_h = entmax(z_h), z_hc = gamma <q_h, kbar_c>/sqrt(d)   =>  dz_h by the Jacobian above
//   dq_h = gamma/sqrt(d) sum_c dz_hc kbar_c (written, fp32);   dkbar_c += gamma/sqrt(d) sum_h dz_hc q_h (atomic, fp32)
// Only routed chunks are touched, SEG list entries at a time.  Margins: eight chunks at once, four lanes per summary row
// (lane l reads the 16-byte pieces (l mod 4) + 4 j of the chunk l div 4, so that a query piece read from shared memory
// serves eight chunks and two shuffles per head finish a dot product); they stay in shared memory until the whole list
// has been seen, which fixes dz.  Then lanes own head_dim slices: dq_h += dz_hc kbar_c, dkbar_c by vector reductions (the L2
// atomic units count requests, not bytes).  8192 tokens, 32/8 heads, chunks of 64: 690 us with two sweeps of butterfly
// reductions over the list, now 435.
//
// summaries_bwd_kernel: four warps per (batch, KV head, chunk), a quarter of its rows each: Eq. 3, kbar_c = sum_t a_t k_t with
// a = softmax(<qbar, k_t>/sqrt(d)) (a_t = 1/B without a summary query): dk_t += a_t dkbar_c + ds_t qbar/sqrt(d),
// ds_t = a_t (<k_t, dkbar_c> - sum_u a_u <k_u, dkbar_c>), dqbar += sum_t ds_t k_t / sqrt(d).  The B logits and products of the
// chunk meet in shared memory.
#include <initializer_list>

#include "common.cuh"

namespace dash {

constexpr int RB_WARPS = 4;

// The fp32 buffers of these two entry points may sit anywhere a float may (a view into a flat gradient buffer): VEC, 16-byte
// accesses, only where all of a call's are 16-byte aligned.
static bool all_aligned16(std::initializer_list<const void*> ptrs) {
  for (const void* p : ptrs)
    if (reinterpret_cast<uintptr_t>(p) & 15) return false;
  return true;
}

__global__ void __launch_bounds__(256) zero_kernel(float* p, long long n, bool vec) {
  chain_wait();
  chain_release();
  const long long thread = (long long)blockIdx.x * 256 + threadIdx.x, threads = (long long)gridDim.x * 256;
  if (vec) {
    zero_floats(p, n, thread, threads);
  } else {
    for (long long k = thread; k < n; k += threads) p[k] = 0.f;
  }
}
static cudaError_t launch_zero(float* p, size_t bytes, cudaStream_t st) {
  const long long n = (long long)(bytes / sizeof(float)), blocks = (n + 1023) / 1024, most = 2 * current_sm_count();
  cudaError_t e = launch_chained(zero_kernel, dim3((unsigned)(blocks < most ? blocks : most)), dim3(256), 0, st, p, n, all_aligned16({p}));
  count_launch();
  return e;
}

// 4 or 2 consecutive floats added to global memory, in one request where they are aligned.
template <int V, bool VEC>
__device__ __forceinline__ void add_global(float* p, const float (&x)[V]) {
  if constexpr (!VEC) {
#pragma unroll
    for (int v = 0; v < V; ++v) atomicAdd(p + v, x[v]);
  } else if constexpr (V == 4)
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]) : "memory");
  else
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(x[0]), "f"(x[1]) : "memory");
}
template <int V, bool VEC = true, typename T>
__device__ __forceinline__ void load_vec(const T* p, float (&x)[V]) {
  if constexpr (!VEC) {
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] = p[v];
  } else if constexpr (V == 4) {
    const float4 f = load4(p);
    x[0] = f.x; x[1] = f.y; x[2] = f.z; x[3] = f.w;
  } else {
    const float2 f = load2(p);
    x[0] = f.x; x[1] = f.y;
  }
}

template <int V, bool VEC>
__device__ __forceinline__ void store_vec(float* p, const float (&x)[V]) {
  if constexpr (!VEC) {
#pragma unroll
    for (int v = 0; v < V; ++v) p[v] = x[v];
  } else if constexpr (V == 4) {
    store4(p, make_float4(x[0], x[1], x[2], x[3]));
  } else {
    *reinterpret_cast<float2*>(p) = make_float2(x[0], x[1]);
  }
}

// G (heads per KV head) is a template parameter so that the per-head sums live in registers.
template <typename T, int D, int G, bool VEC>
__global__ void __launch_bounds__(RB_WARPS * 32, G > 4 ? 1 : D == 128 ? 5 : 7)
route_bwd_kernel(Dims dm, const T* __restrict__ Q, const float* __restrict__ Kbar, const int* __restrict__ count,
                 const int* __restrict__ blk_idx, const float* __restrict__ tau, const float* __restrict__ dbias,
                 float* __restrict__ dQr, float* __restrict__ dKbar) {
  constexpr int VPL = D / 32;
  constexpr int SEG = G <= 8 ? 64 : 32;        // list entries held at a time
  __shared__ __align__(16) float q_s[RB_WARPS][G][D];
  __shared__ __align__(16) float m_s[RB_WARPS][SEG][G];      // margins, then dz
  __shared__ float dw_s[RB_WARPS][SEG];
  __shared__ int c_s[RB_WARPS][SEG];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long gw = (long long)blockIdx.x * RB_WARPS + warp;
  const long long total = (long long)dm.batch * dm.h_kv * dm.seq_q;
  chain_wait();
  chain_release();
  if (gw >= total) return;
  const int i = (int)(gw % dm.seq_q);
  const long long grp = gw / dm.seq_q;
  const int r = (int)(grp % dm.h_kv), b = (int)(grp / dm.h_kv);
  // fp32 gradient of Q from the routing: [batch, seq_q, h_q, d], every row written (zeros where nothing is routed)
  float* dq_out = dQr + (((long long)b * dm.seq_q + i) * dm.h_q + (long long)r * G) * D + lane * VPL;
  const int c_own = i >> dm.log_b;
  const int n_local = min(dm.local_blocks, c_own);              // window chunks close the list and carry no gradient
  const int n_routed = count[grp * dm.seq_q + i] - n_local;
  // (pairs of floats: one instruction for two products)
  float2 dq[G][VPL / 2];
#pragma unroll
  for (int h = 0; h < G; ++h)
#pragma unroll
    for (int v = 0; v < VPL / 2; ++v) dq[h][v] = make_float2(0.f, 0.f);
  if (n_routed > 0) {
    const long long loff = grp * dm.list_rows + list_row_offset(dm, i);
    const float* kb = Kbar + grp * dm.T_s * D;
    // the queries stay in registers for the second part where those suffice (shared memory costs four wavefronts a read)
    constexpr bool Q_REGS = G <= 4;
    [[maybe_unused]] float qr[Q_REGS ? G : 1][VPL];
    float th[G];
#pragma unroll
    for (int h = 0; h < G; ++h) {
      float x[VPL];
      load_vec<VPL>(Q + (long long)b * dm.qs[0] + (long long)i * dm.qs[1] + (long long)(r * G + h) * dm.qs[2] + lane * VPL, x);
#pragma unroll
      for (int v = 0; v < VPL; ++v) {
        q_s[warp][h][lane * VPL + v] = x[v];
        if (Q_REGS) qr[Q_REGS ? h : 0][v] = x[v];
      }
      th[h] = tau[((long long)b * dm.h_q + r * G + h) * dm.seq_q + i];
    }
    float dmean = 0.f;
    for (int k = lane; k < n_routed; k += 32) dmean += dbias[loff + k];
    dmean = warp_sum(dmean) / (float)n_routed;
    const float e = dm.e;
    const int e_int = dm.e_int;
    float A[G], S[G];                          // per head A_h = sum_c s_hc dw_c / g_q and S_h = sum_c s_hc
#pragma unroll
    for (int h = 0; h < G; ++h) A[h] = S[h] = 0.f;
    // Margins m_hc = x_scale <q_h, kbar_c> - tau_h (clamped at 0) and weight gradients dw_c of entries [k0, k0 + n)
    auto margins = [&](int k0, int n, bool sum) {
      __syncwarp();
      for (int k = lane; k < n; k += 32) {
        c_s[warp][k] = blk_idx[loff + k0 + k];
        dw_s[warp][k] = (dbias[loff + k0 + k] - dmean) * dm.inv_sigma;
      }
      __syncwarp();
      for (int e0 = 0; e0 < n; e0 += 8) {
        const int k = e0 + (lane >> 2);
        const bool live = k < n;
        const float* kp = kb + (long long)c_s[warp][min(k, n - 1)] * D + 4 * (lane & 3);
        float x[G];
        {
          float2 xp[G];
#pragma unroll
          for (int h = 0; h < G; ++h) xp[h] = make_float2(0.f, 0.f);
          float4 kv[D / 16];
#pragma unroll
          for (int j = 0; j < D / 16; ++j)
            kv[j] = VEC ? load4(kp + 16 * j) : make_float4(kp[16 * j], kp[16 * j + 1], kp[16 * j + 2], kp[16 * j + 3]);
#pragma unroll
          for (int j = 0; j < D / 16; ++j)
#pragma unroll
            for (int h = 0; h < G; ++h) {
              const float4 qv = load4(&q_s[warp][h][16 * j + 4 * (lane & 3)]);
              xp[h] = __ffma2_rn(make_float2(qv.x, qv.y), make_float2(kv[j].x, kv[j].y), xp[h]);
              xp[h] = __ffma2_rn(make_float2(qv.z, qv.w), make_float2(kv[j].z, kv[j].w), xp[h]);
            }
#pragma unroll
          for (int h = 0; h < G; ++h) x[h] = xp[h].x + xp[h].y;
        }
        float w = 0.f;
#pragma unroll
        for (int h = 0; h < G; ++h) {
          x[h] += __shfl_xor_sync(0xffffffffu, x[h], 1);
          x[h] += __shfl_xor_sync(0xffffffffu, x[h], 2);
          x[h] = fmaxf(x[h] * dm.x_scale - th[h], 0.f);
          w += pow_e(x[h], e_int, e);
        }
        w /= (float)G;
        const float dw = live && w > 0.f ? dw_s[warp][k] / (w * (float)G) : 0.f;
        if (live && sum) {
#pragma unroll
          for (int h = 0; h < G; ++h) {
            const float s = pow_em1(x[h], e_int, e);
            A[h] = fmaf(s, dw, A[h]);
            S[h] += s;
          }
        }
        __syncwarp();                           // (everybody has read dw_s of these entries)
        if (live && (lane & 3) == 0) {
          dw_s[warp][k] = dw;                   // from here on the gradient w.r.t. every head's weight
#pragma unroll
          for (int h = 0; h < G; ++h) m_s[warp][k][h] = x[h];
        }
      }
      __syncwarp();
    };
    for (int k0 = 0; k0 < n_routed; k0 += SEG) margins(k0, min(SEG, n_routed - k0), true);
    // (the four lanes of a chunk hold the same sums)
#pragma unroll
    for (int o = 4; o < 32; o <<= 1)
#pragma unroll
      for (int h = 0; h < G; ++h) {
        A[h] += __shfl_xor_sync(0xffffffffu, A[h], o);
        S[h] += __shfl_xor_sync(0xffffffffu, S[h], o);
      }
    const float zscale = dm.x_scale / (1.f / e);       // gamma / sqrt(d) = x_scale / (alpha - 1)
#pragma unroll
    for (int h = 0; h < G; ++h) A[h] = S[h] > 0.f ? A[h] / S[h] : 0.f;
    for (int k0 = 0; k0 < n_routed; k0 += SEG) {
      const int n = min(SEG, n_routed - k0);
      if (n_routed > SEG) margins(k0, n, false);
      // dz_hc = s_hc (dw_c / g_q - A_h / S_h), scaled
      for (int k = lane; k < n; k += 32) {
        const float dw = dw_s[warp][k];
#pragma unroll
        for (int h = 0; h < G; ++h)
          m_s[warp][k][h] = S[h] > 0.f ? pow_em1(m_s[warp][k][h], e_int, e) * (dw - A[h]) * zscale : 0.f;
      }
      __syncwarp();
      constexpr int NB = 4;
      for (int e0 = 0; e0 < n; e0 += NB) {
        float kv[NB][VPL];
        int c[NB];
#pragma unroll
        for (int u = 0; u < NB; ++u) {
          c[u] = c_s[warp][min(e0 + u, n - 1)];
          load_vec<VPL, VEC>(kb + (long long)c[u] * D + lane * VPL, kv[u]);
        }
#pragma unroll
        for (int u = 0; u < NB; ++u) {
          if (e0 + u < n) {
            float2 dkb[VPL / 2];
#pragma unroll
            for (int v = 0; v < VPL / 2; ++v) dkb[v] = make_float2(0.f, 0.f);
#pragma unroll
            for (int h = 0; h < G; ++h) {
              const float dz = m_s[warp][e0 + u][h];
              const float2 dz2 = make_float2(dz, dz);
              [[maybe_unused]] float qs[VPL];
              if constexpr (!Q_REGS) load_vec<VPL>(&q_s[warp][h][lane * VPL], qs);
#pragma unroll
              for (int v = 0; v < VPL / 2; ++v) {
                const float2 qv = Q_REGS ? make_float2(qr[Q_REGS ? h : 0][2 * v], qr[Q_REGS ? h : 0][2 * v + 1]) : make_float2(qs[2 * v], qs[2 * v + 1]);
                dq[h][v] = __ffma2_rn(dz2, make_float2(kv[u][2 * v], kv[u][2 * v + 1]), dq[h][v]);
                dkb[v] = __ffma2_rn(dz2, qv, dkb[v]);
              }
            }
            float out[VPL];
#pragma unroll
            for (int v = 0; v < VPL / 2; ++v) { out[2 * v] = dkb[v].x; out[2 * v + 1] = dkb[v].y; }
            add_global<VPL, VEC>(dKbar + (grp * dm.T_s + c[u]) * D + lane * VPL, out);
          }
        }
      }
    }
  }
#pragma unroll
  for (int h = 0; h < G; ++h) {
    float x[VPL];
#pragma unroll
    for (int v = 0; v < VPL / 2; ++v) { x[2 * v] = dq[h][v].x; x[2 * v + 1] = dq[h][v].y; }
    store_vec<VPL, VEC>(dq_out + (long long)h * D, x);
  }
}

// The same for sixteen consecutive tokens per block, a warp each, whose lists fit in shared memory together: dz stays there, and
// once all sixteen are done the block goes through the chunks that any of them routed, one warp per chunk, and sends one
// reduction per chunk instead of one per token and chunk.  The reductions were what bounded the kernel above: the L2's atomic
// units take about 97 G requests a second whatever their width, and 8192 tokens, 32/8 heads, chunks of 64 send 36 M of them.
constexpr int RT_TOK = 16;
template <int G>
struct RouteTile {      // offsets in dynamic shared memory, for lists of up to `cap` chunks (a multiple of 8)
  static constexpr size_t ENTRY = 4 * G + 4 + 2 + 2;      // margin or dz per head, dw, chunk id, place of a chunk in the list
  __host__ __device__ static size_t bytes(int cap, int d, int elem) { return (size_t)RT_TOK * cap * ENTRY + (size_t)RT_TOK * G * d * elem + (size_t)cap * 4; }
};

template <typename T, int D, int G, bool VEC>
__global__ void __launch_bounds__(RT_TOK * 32, 2)
route_bwd_tile_kernel(Dims dm, const T* __restrict__ Q, const float* __restrict__ Kbar, const int* __restrict__ count,
                      const int* __restrict__ blk_idx, const float* __restrict__ tau, const float* __restrict__ dbias,
                      float* __restrict__ dQr, float* __restrict__ dKbar, int n_tiles, int cap) {
  constexpr int VPL = D / 32;
  extern __shared__ __align__(16) uint8_t smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* m_all = reinterpret_cast<float*>(smem);                                  // [token][cap][G]
  T* q_all = reinterpret_cast<T*>(m_all + (size_t)RT_TOK * cap * G);              // [token][G][D]
  float* dw_s = reinterpret_cast<float*>(q_all + RT_TOK * G * D) + warp * cap;    // [token][cap]
  uint32_t* bits_s = reinterpret_cast<uint32_t*>(dw_s - warp * cap + RT_TOK * cap);      // [cap]: the tokens that routed a chunk
  unsigned short* c_s = reinterpret_cast<unsigned short*>(bits_s + cap) + warp * cap;    // [token][cap]
  unsigned short* pos_all = c_s - warp * cap + RT_TOK * cap;                      // [token][cap]
  float* m_s = m_all + (size_t)warp * cap * G;
  T* q_s = q_all + warp * G * D;
  for (int c = threadIdx.x; c < cap; c += RT_TOK * 32) bits_s[c] = 0u;
  chain_wait();
  chain_release();
  __syncthreads();
  const long long grp = blockIdx.x / n_tiles;
  const int i0 = (int)(blockIdx.x % n_tiles) * RT_TOK, i = i0 + warp;
  const int r = (int)(grp % dm.h_kv), b = (int)(grp / dm.h_kv);
  const float* kb = Kbar + grp * dm.T_s * D;
  const int c_own = i >> dm.log_b;
  const int n_routed = i < dm.seq_q ? count[grp * dm.seq_q + i] - min(dm.local_blocks, c_own) : 0;      // (window chunks close the list)
  const float e = dm.e;
  const int e_int = dm.e_int;
  float2 dq[G][VPL / 2];
#pragma unroll
  for (int h = 0; h < G; ++h)
#pragma unroll
    for (int v = 0; v < VPL / 2; ++v) dq[h][v] = make_float2(0.f, 0.f);
  if (n_routed > 0) {
    const long long loff = grp * dm.list_rows + list_row_offset(dm, i);
    float th[G];
#pragma unroll
    for (int h = 0; h < G; ++h) {
      const T* qp = Q + (long long)b * dm.qs[0] + (long long)i * dm.qs[1] + (long long)(r * G + h) * dm.qs[2] + lane * VPL;
      if constexpr (VPL == 4 && sizeof(T) == 2) *reinterpret_cast<uint2*>(q_s + h * D + lane * VPL) = *reinterpret_cast<const uint2*>(qp);
      else
#pragma unroll
        for (int v = 0; v < VPL; ++v) q_s[h * D + lane * VPL + v] = qp[v];
      th[h] = tau[((long long)b * dm.h_q + r * G + h) * dm.seq_q + i];
    }
    float dmean = 0.f;
    for (int k = lane; k < n_routed; k += 32) {
      const int c = blk_idx[loff + k];
      const float db = dbias[loff + k];
      c_s[k] = (unsigned short)c;
      pos_all[warp * cap + c] = (unsigned short)k;
      atomicOr(&bits_s[c], 1u << warp);
      dw_s[k] = db;
      dmean += db;
    }
    dmean = warp_sum(dmean) / (float)n_routed;
    __syncwarp();
    // margins, eight chunks at once (as above)
    float A[G], S[G];
#pragma unroll
    for (int h = 0; h < G; ++h) A[h] = S[h] = 0.f;
#pragma unroll 1
    for (int e0 = 0; e0 < n_routed; e0 += 8) {
      const int k = e0 + (lane >> 2);
      const bool live = k < n_routed;
      const float* kp = kb + (long long)c_s[min(k, n_routed - 1)] * D + 4 * (lane & 3);
      float2 xp[G];
#pragma unroll
      for (int h = 0; h < G; ++h) xp[h] = make_float2(0.f, 0.f);
      float4 kv[D / 16];
#pragma unroll
      for (int j = 0; j < D / 16; ++j)
        kv[j] = VEC ? load4(kp + 16 * j) : make_float4(kp[16 * j], kp[16 * j + 1], kp[16 * j + 2], kp[16 * j + 3]);
#pragma unroll
      for (int j = 0; j < D / 16; ++j)
#pragma unroll
        for (int h = 0; h < G; ++h) {
          const float4 qv = load4(q_s + h * D + 16 * j + 4 * (lane & 3));
          xp[h] = __ffma2_rn(make_float2(qv.x, qv.y), make_float2(kv[j].x, kv[j].y), xp[h]);
          xp[h] = __ffma2_rn(make_float2(qv.z, qv.w), make_float2(kv[j].z, kv[j].w), xp[h]);
        }
      float x[G], w = 0.f;
#pragma unroll
      for (int h = 0; h < G; ++h) {
        x[h] = xp[h].x + xp[h].y;
        x[h] += __shfl_xor_sync(0xffffffffu, x[h], 1);
        x[h] += __shfl_xor_sync(0xffffffffu, x[h], 2);
        x[h] = fmaxf(x[h] * dm.x_scale - th[h], 0.f);
        w += pow_e(x[h], e_int, e);
      }
      w /= (float)G;
      const float dw = live && w > 0.f ? (dw_s[k] - dmean) * dm.inv_sigma / (w * (float)G) : 0.f;
      __syncwarp();                           // (everybody has read dw_s of these entries)
      if (live) {
#pragma unroll
        for (int h = 0; h < G; ++h) {
          const float sp = pow_em1(x[h], e_int, e);
          A[h] = fmaf(sp, dw, A[h]);
          S[h] += sp;
        }
        if ((lane & 3) == 0) {
          dw_s[k] = dw;                       // from here on the gradient w.r.t. every head's weight
#pragma unroll
          for (int h = 0; h < G; ++h) m_s[k * G + h] = x[h];
        }
      }
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1)
#pragma unroll
      for (int h = 0; h < G; ++h) {
        A[h] += __shfl_xor_sync(0xffffffffu, A[h], o);
        S[h] += __shfl_xor_sync(0xffffffffu, S[h], o);
      }
    const float zscale = dm.x_scale / (1.f / e);       // gamma / sqrt(d) = x_scale / (alpha - 1)
#pragma unroll
    for (int h = 0; h < G; ++h) A[h] = S[h] > 0.f ? A[h] / S[h] : 0.f;
    __syncwarp();
    // dz_hc = s_hc (dw_c / g_q - A_h / S_h), scaled
    for (int k = lane; k < n_routed; k += 32) {
      const float dw = dw_s[k];
#pragma unroll
      for (int h = 0; h < G; ++h)
        m_s[k * G + h] = S[h] > 0.f ? pow_em1(m_s[k * G + h], e_int, e) * (dw - A[h]) * zscale : 0.f;
    }
    __syncwarp();
    constexpr int NB = 4;
#pragma unroll 1
    for (int e0 = 0; e0 < n_routed; e0 += NB) {
      float kv[NB][VPL];
#pragma unroll
      for (int u = 0; u < NB; ++u) load_vec<VPL, VEC>(kb + (long long)c_s[min(e0 + u, n_routed - 1)] * D + lane * VPL, kv[u]);
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        if (e0 + u < n_routed) {
#pragma unroll
          for (int h = 0; h < G; ++h) {
            const float dz = m_s[(e0 + u) * G + h];
#pragma unroll
            for (int v = 0; v < VPL / 2; ++v) dq[h][v] = __ffma2_rn(make_float2(dz, dz), make_float2(kv[u][2 * v], kv[u][2 * v + 1]), dq[h][v]);
          }
        }
      }
    }
  }
  if (i < dm.seq_q) {
    float* dq_out = dQr + (((long long)b * dm.seq_q + i) * dm.h_q + (long long)r * G) * D + lane * VPL;
#pragma unroll
    for (int h = 0; h < G; ++h) {
      float x[VPL];
#pragma unroll
      for (int v = 0; v < VPL / 2; ++v) { x[2 * v] = dq[h][v].x; x[2 * v + 1] = dq[h][v].y; }
      store_vec<VPL, VEC>(dq_out + (long long)h * D, x);
    }
  }
  __syncthreads();
  // dkbar of the chunks that any of the block's tokens routed
  const int n_c = min(min(i0 + RT_TOK, dm.seq_q) - 1 >> dm.log_b, dm.T_s);
#pragma unroll 1
  for (int c = warp; c < n_c; c += RT_TOK) {
    uint32_t bits = bits_s[c];
    if (bits == 0u) continue;
    float2 dkb[VPL / 2];
#pragma unroll
    for (int v = 0; v < VPL / 2; ++v) dkb[v] = make_float2(0.f, 0.f);
    while (bits) {
      const int t = __ffs(bits) - 1;
      bits &= bits - 1;
      const float* dz = m_all + ((size_t)t * cap + pos_all[t * cap + c]) * G;
      const T* qp = q_all + t * G * D + lane * VPL;
#pragma unroll
      for (int h = 0; h < G; ++h) {
        float q[VPL];
        load_vec<VPL>(qp + h * D, q);
#pragma unroll
        for (int v = 0; v < VPL / 2; ++v) dkb[v] = __ffma2_rn(make_float2(dz[h], dz[h]), make_float2(q[2 * v], q[2 * v + 1]), dkb[v]);
      }
    }
    float out[VPL];
#pragma unroll
    for (int v = 0; v < VPL / 2; ++v) { out[2 * v] = dkb[v].x; out[2 * v + 1] = dkb[v].y; }
    add_global<VPL, VEC>(dKbar + (grp * dm.T_s + c) * D + lane * VPL, out);
  }
}

constexpr int SB_SPLIT = 4;      // warps that share a chunk = a block

template <typename T, int D, bool VEC>
__global__ void __launch_bounds__(SB_SPLIT * 32)
summaries_bwd_kernel(Dims dm, const T* __restrict__ K, const float* __restrict__ qbar, long long qbar_chunk_stride,
                     const float* __restrict__ dKbar, float* __restrict__ dK, float* __restrict__ dqbar) {
  constexpr int VPL = D / 32, NB = 4;
  __shared__ float s_s[128], da_s[128];      // logits and <k_t, dkbar> of the chunk's tokens
  __shared__ float red[SB_SPLIT][D];
  chain_wait();
  chain_release();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = (int)(blockIdx.x % dm.T_s);
  const long long grp = blockIdx.x / dm.T_s;
  const int r = (int)(grp % dm.h_kv), b = (int)(grp / dm.h_kv);
  const int rows = dm.B / SB_SPLIT, t0 = warp * rows;          // this warp's tokens of the chunk (4 .. 32)
  const T* kp = K + (long long)b * dm.ks[0] + (long long)c * dm.B * dm.ks[1] + (long long)r * dm.ks[2] + lane * VPL;
  float* dkp = dK + (((long long)b * dm.seq_kv + (long long)c * dm.B) * dm.h_kv + r) * D + lane * VPL;
  const long long gtok = (long long)dm.h_kv * D;
  float g[VPL];
  load_vec<VPL, VEC>(dKbar + (grp * dm.T_s + c) * D + lane * VPL, g);
  // dk rows of four tokens at a time: read, add, write
  auto add_rows = [&](int t, auto&& delta) {
    float x[NB][VPL];
#pragma unroll
    for (int u = 0; u < NB; ++u) load_vec<VPL, VEC>(dkp + (long long)(t + u) * gtok, x[u]);
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      delta(u, x[u]);
      store_vec<VPL, VEC>(dkp + (long long)(t + u) * gtok, x[u]);
    }
  };
  if (qbar == nullptr) {
    const float inv = 1.f / (float)dm.B;
    for (int t = t0; t < t0 + rows; t += NB)
      add_rows(t, [&](int, float (&x)[VPL]) {
#pragma unroll
        for (int v = 0; v < VPL; ++v) x[v] = fmaf(g[v], inv, x[v]);
      });
    return;
  }
  float qv[VPL];
  load_vec<VPL, VEC>(qbar + (long long)c * qbar_chunk_stride + (long long)r * D + lane * VPL, qv);
  for (int t = t0; t < t0 + rows; t += NB) {
    float kv[NB][VPL], s[NB], da[NB];
#pragma unroll
    for (int u = 0; u < NB; ++u) load_vec<VPL>(kp + (long long)(t + u) * dm.ks[1], kv[u]);
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      s[u] = da[u] = 0.f;
#pragma unroll
      for (int v = 0; v < VPL; ++v) {
        s[u] = fmaf(qv[v], kv[u][v], s[u]);
        da[u] = fmaf(g[v], kv[u][v], da[u]);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
        da[u] += __shfl_xor_sync(0xffffffffu, da[u], o);
      }
#pragma unroll
    for (int u = 0; u < NB; ++u)
      if (lane == u) { s_s[t + u] = s[u] * dm.sm_scale; da_s[t + u] = da[u]; }
  }
  __syncthreads();
  // softmax statistics and sum_t a_t <k_t, g>, by every warp for itself
  float mx = -INFINITY, l = 0.f, ada = 0.f;
  for (int t = lane; t < dm.B; t += 32) mx = fmaxf(mx, s_s[t]);
  mx = warp_max(mx);
  for (int t = lane; t < dm.B; t += 32) {
    const float p = __expf(s_s[t] - mx);
    l += p;
    ada = fmaf(p, da_s[t], ada);
  }
  const float inv_l = 1.f / warp_sum(l);
  ada = warp_sum(ada) * inv_l;
  float dqb[VPL];
#pragma unroll
  for (int v = 0; v < VPL; ++v) dqb[v] = 0.f;
  for (int t = t0; t < t0 + rows; t += NB) {
    float kv[NB][VPL];
#pragma unroll
    for (int u = 0; u < NB; ++u) load_vec<VPL>(kp + (long long)(t + u) * dm.ks[1], kv[u]);
    add_rows(t, [&](int u, float (&x)[VPL]) {
      const float a = __expf(s_s[t + u] - mx) * inv_l, dst = a * (da_s[t + u] - ada);
#pragma unroll
      for (int v = 0; v < VPL; ++v) {
        x[v] += a * g[v] + dst * qv[v] * dm.sm_scale;
        dqb[v] = fmaf(dst, kv[u][v], dqb[v]);
      }
    });
  }
  if (dqbar) {
#pragma unroll
    for (int v = 0; v < VPL; ++v) red[warp][lane * VPL + v] = dqb[v] * dm.sm_scale;
    __syncthreads();
    if (warp == 0) {
#pragma unroll
      for (int v = 0; v < VPL; ++v)
        dqb[v] = (red[0][lane * VPL + v] + red[1][lane * VPL + v]) + (red[2][lane * VPL + v] + red[3][lane * VPL + v]);
      add_global<VPL, VEC>(dqbar + (long long)c * qbar_chunk_stride + (long long)r * D + lane * VPL, dqb);
    }
  }
}

// Tiles of sixteen tokens: causal lists (no longer than T_s, and the tokens of a tile share their own chunk) of groups of up to
// eight heads, where two blocks fit on an SM (bf16, four heads, d 128: up to 184 chunks).  Longer lists take a warp per row.
static int route_tile_cap(const Dims& dm) { return (dm.T_s + 7) / 8 * 8; }
template <typename T, int D, int G>
static bool tiles_fit(const Dims& dm) {
  return dm.causal && G <= 8 && RouteTile<G>::bytes(route_tile_cap(dm), D, sizeof(T)) <= 112 * 1024;
}
template <typename T, int D, int G, bool VEC>
static cudaError_t launch_route_tiles(const Dims& dm, const T* Q, const float* Kbar, const int* count, const int* blk_idx,
                                      const float* tau, const float* dbias, float* dQr, float* dKbar, cudaStream_t st) {
  if constexpr (G > 8) {
    return cudaErrorInvalidValue;
  } else {
    static std::atomic<unsigned long long> configured{0};
    auto kern = route_bwd_tile_kernel<T, D, G, VEC>;
    if (cudaError_t e = allow_dynamic_smem(kern, 112 * 1024, configured); e != cudaSuccess) return e;
    const int n_tiles = (dm.seq_q + RT_TOK - 1) / RT_TOK, cap = route_tile_cap(dm);
    return launch_chained(kern, dim3((unsigned)((long long)dm.batch * dm.h_kv * n_tiles)), dim3(RT_TOK * 32),
                          RouteTile<G>::bytes(cap, D, sizeof(T)), st, dm, Q, Kbar, count, blk_idx, tau, dbias, dQr, dKbar, n_tiles, cap);
  }
}

cudaError_t launch_route_bwd(const Dims& dm, const void* Q, const float* Kbar, const int* count, const int* blk_idx,
                             const float* tau, const float* dbias, float* dQr, float* dKbar, cudaStream_t st) {
  const size_t kb_bytes = (size_t)dm.batch * dm.h_kv * (size_t)dm.T_s * dm.d * sizeof(float);
  if (kb_bytes > 0) {
    cudaError_t e = launch_zero(dKbar, kb_bytes, st);
    if (e != cudaSuccess) return e;
  }
  const long long total = (long long)dm.batch * dm.h_kv * dm.seq_q;
  const unsigned grid = (unsigned)((total + RB_WARPS - 1) / RB_WARPS);
  cudaError_t le = cudaSuccess;
  const bool vec = all_aligned16({Kbar, dQr, dKbar});
#define DASH_RB_V(T, D, GV, V) \
  le = launch_chained(route_bwd_kernel<T, D, GV, V>, dim3(grid), dim3(RB_WARPS * 32), 0, st, dm, (const T*)Q, Kbar, count, blk_idx, tau, dbias, dQr, dKbar)
#define DASH_RB(T, D, GV) \
  if (tiles_fit<T, D, GV>(dm)) \
    le = vec ? launch_route_tiles<T, D, GV, true>(dm, (const T*)Q, Kbar, count, blk_idx, tau, dbias, dQr, dKbar, st) \
             : launch_route_tiles<T, D, GV, false>(dm, (const T*)Q, Kbar, count, blk_idx, tau, dbias, dQr, dKbar, st); \
  else if (vec) DASH_RB_V(T, D, GV, true); else DASH_RB_V(T, D, GV, false)
#define DASH_RB_G(T, D)                   \
  switch (dm.g_q) {                       \
    case 1: DASH_RB(T, D, 1); break;      \
    case 2: DASH_RB(T, D, 2); break;      \
    case 4: DASH_RB(T, D, 4); break;      \
    case 8: DASH_RB(T, D, 8); break;      \
    case 16: DASH_RB(T, D, 16); break;    \
    default: return cudaErrorInvalidValue; \
  }
  if (dm.dtype == DASH_BF16) {
    if (dm.d == 128) { DASH_RB_G(__nv_bfloat16, 128) } else { DASH_RB_G(__nv_bfloat16, 64) }
  } else {
    if (dm.d == 128) { DASH_RB_G(float, 128) } else { DASH_RB_G(float, 64) }
  }
#undef DASH_RB_G
#undef DASH_RB
#undef DASH_RB_V
  count_launch();
  return le;
}

cudaError_t launch_summaries_bwd(const Dims& dm, const void* K, const float* qbar, long long qbar_chunk_stride,
                                 const float* dKbar, float* dK, float* dqbar, size_t dqbar_bytes, cudaStream_t st) {
  if (dqbar && dqbar_bytes > 0) {
    cudaError_t e = launch_zero(dqbar, dqbar_bytes, st);
    if (e != cudaSuccess) return e;
  }
  const long long total = (long long)dm.batch * dm.h_kv * dm.T_s;
  if (total == 0) return cudaSuccess;
  const unsigned grid = (unsigned)total;
  cudaError_t le = cudaSuccess;
  const bool vec = all_aligned16({qbar, dKbar, dK, dqbar});
#define DASH_SB_V(T, D, V) \
  le = launch_chained(summaries_bwd_kernel<T, D, V>, dim3(grid), dim3(SB_SPLIT * 32), 0, st, dm, (const T*)K, qbar, qbar_chunk_stride, dKbar, dK, dqbar)
#define DASH_SB(T, D) \
  do { if (vec) DASH_SB_V(T, D, true); else DASH_SB_V(T, D, false); } while (0)
  if (dm.dtype == DASH_BF16) {
    if (dm.d == 128) DASH_SB(__nv_bfloat16, 128); else DASH_SB(__nv_bfloat16, 64);
  } else {
    if (dm.d == 128) DASH_SB(float, 128); else DASH_SB(float, 64);
  }
#undef DASH_SB
#undef DASH_SB_V
  count_launch();
  return le;
}

}  // namespace dash
