// Leaf recurrence for layers whose weights fit the shared memory of ONE cluster (fp32 up to d = 256, bf16 up to d = 384 with
// d_ff = 4 d): the sequential part of Algorithm 1 for the positions [t0, t1) of one leaf.
//
// The sequences are independent (Sec. 2.2 states the layer per sequence), so a cluster of 16 CTAs takes one to three of them
// and clusters never talk to each other.  Inside a cluster a token step is the usual chain of five small all-to-all
// exchanges, but through distributed shared memory: every vector has a copy in each CTA, the warp that finishes rows of it
// sends them to all 16 copies with st.async, and the stores count themselves into the receiver's mbarrier.  No flags, no
// polling of L2, no barrier across warps: a warp waits for the vector's mbarrier, multiplies its own rows (lanes over K,
// sums by shuffles, weights in shared memory for the whole launch) and sends.  Exchanged values stay fp32.
// A buffer is written again only a whole step later, and everything a step writes depends, through the chain, on every
// warp having read what the step before left there, so one copy of each vector is enough.
// What bounds it: five hops of about half a microsecond; the arithmetic of a step is a few hundred cycles.
#include <cuda_bf16.h>
#include <string.h>

#include <type_traits>

#include "rt_handover.h"
#include "rt_kernels.h"
#include "rt_tc.cuh"

namespace rt {

namespace {

constexpr int kCl = 16;                           // CTAs per cluster
constexpr int kSmWarps = 16;                      // mat-vec warps per CTA; then one attention warp on the chain and four beside it
constexpr int kFoldWarps = 4;                     // two lanes per query of the leaf: 64 queries
constexpr int kSmThreads = (kSmWarps + 1 + kFoldWarps) * 32;
constexpr int kSmLeafMax = kFoldWarps * 16;
constexpr int kFin = Handover::kSlots;            // final (k, v) of the last four positions
constexpr int kStateStride = kHeadDim + 4;        // o[64], m, l of the query that is finished next

struct SmallLayout {
  unsigned off_c, off_h, off_g, off_z, off_kv, off_gain, off_fin, off_st, off_wo, off_wup, off_wdn, off_wk, off_wv, total;
};

SmallLayout small_layout(size_t es, int nb, int d, int dff) {
  SmallLayout L;
  size_t o = 160;                                 // abort flag, mbarriers
  auto take = [&](size_t n) { const size_t at = o; o += align_up(n, 16); return (unsigned)at; };
  L.off_c = take((size_t)nb * d * 4); L.off_h = take((size_t)nb * d * 4); L.off_z = take((size_t)nb * d * 4);
  L.off_g = take((size_t)nb * dff * 4);
  L.off_kv = take(2 * kHeadDim * 4);              // raw k, v of the pair this CTA owns
  L.off_gain = take((size_t)2 * d * 4);
  L.off_fin = take((size_t)kFin * 2 * kHeadDim * 4);
  L.off_st = take((size_t)2 * kStateStride * 4);
  const size_t wd = (size_t)(d / kCl) * d * es, wf = (size_t)(dff / kCl) * d * es;
  L.off_wo = take(wd); L.off_wup = take(wf); L.off_wdn = take(wf); L.off_wk = take(wd); L.off_wv = take(wd);
  L.total = (unsigned)o;
  return L;
}

__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_arrive_wait() {
  asm volatile("barrier.cluster.arrive.aligned;\n barrier.cluster.wait.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_to(uint32_t addr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Remote stores that add their bytes to the receiver's mbarrier.
__device__ __forceinline__ void send(uint32_t dst, uint32_t bar, const float (&v)[1]) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(dst), "r"(__float_as_uint(v[0])), "r"(bar) : "memory");
}
__device__ __forceinline__ void send(uint32_t dst, uint32_t bar, const float (&v)[2]) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1,%2}, [%3];"
               ::"r"(dst), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(bar) : "memory");
}
__device__ __forceinline__ void send(uint32_t dst, uint32_t bar, const float (&v)[4]) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1,%2,%3,%4}, [%5];"
               ::"r"(dst), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])), "r"(bar) : "memory");
}

// Bounded wait of a whole warp that also leaves when another CTA has given up; the answer is the same in every lane.
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int* s_abort, SyncArea* sync) {
  unsigned spins = 0;
  unsigned long long t_start = 0;
  bool ok = true;
  while (ok && !mbar_try_wait_cluster(bar, parity)) {
    if ((++spins & 255u) != 0u) continue;
    if (*s_abort || *reinterpret_cast<volatile unsigned*>(&sync->abort_flag)) { *s_abort = 1; ok = false; break; }
    const unsigned long long now = globaltimer_ns();
    if (t_start == 0) t_start = now;
    else if (now - t_start > kWaitLimitNs) {
      *s_abort = 1;
      sync->status = RT_ERR_TIMEOUT;
      __threadfence();
      atomicExch(&sync->abort_flag, 1u);
      ok = false;
    }
  }
  return __all_sync(0xffffffffu, ok);
}

// U consecutive rows of W (row stride K) times the NB vectors at `vec` ([NB][K] fp32): y[u][b], summed over the warp; with
// SSQ also the sum of squares of each (unscaled) vector.
template <typename T, int U, int NB, bool SSQ>
__device__ __forceinline__ void rows_dot(const T* W, const float* vec, int K, const float* gain, int lane, float (&y)[U][NB], float (&ssq)[NB]) {
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    ssq[b] = 0.f;
#pragma unroll
    for (int u = 0; u < U; ++u) y[u][b] = 0.f;
  }
#pragma unroll 4
  for (int k = lane * 4; k < K; k += 128) {
    float wf[U][4];
#pragma unroll
    for (int u = 0; u < U; ++u) reinterpret_cast<const Vec4<T>*>(W + (size_t)u * K + k)->to_float(wf[u]);
    float4 gn = make_float4(1.f, 1.f, 1.f, 1.f);
    if (SSQ && gain) gn = *reinterpret_cast<const float4*>(gain + k);
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      float4 a = *reinterpret_cast<const float4*>(vec + (size_t)b * K + k);
      if (SSQ) {
        ssq[b] += (a.x * a.x + a.y * a.y) + (a.z * a.z + a.w * a.w);
        a.x *= gn.x; a.y *= gn.y; a.z *= gn.z; a.w *= gn.w;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) y[u][b] += (a.x * wf[u][0] + a.y * wf[u][1]) + (a.z * wf[u][2] + a.w * wf[u][3]);
    }
  }
#pragma unroll
  for (int off = 16; off; off >>= 1) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      if (SSQ) ssq[b] += __shfl_xor_sync(0xffffffffu, ssq[b], off);
#pragma unroll
      for (int u = 0; u < U; ++u) y[u][b] += __shfl_xor_sync(0xffffffffu, y[u][b], off);
    }
  }
}

// TIMERS is compile-time: carried along unused, the stamps cost 5 % of a step.
template <typename T, int NB, bool TIMERS>
__global__ void __launch_bounds__(kSmThreads, 1) leaf_small_kernel(const LeafParams p, const SmallLayout L) {
  extern __shared__ __align__(128) unsigned char smem[];
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem);
  const uint32_t bars = smem_u32(smem + 16);
  const uint32_t bar_c = bars, bar_h = bars + 8, bar_g = bars + 16, bar_z = bars + 24, bar_kv = bars + 32, bar_w = bars + 40;
  // attention: state of query (even, odd) ready; key (mod 4) ready, folded (rt_handover.h)
  const uint32_t bar_state = bars + 48, bar_key = bars + 64, bar_done = bar_key + 8 * Handover::kReadyBars;
  float *vec_c = reinterpret_cast<float*>(smem + L.off_c), *vec_h = reinterpret_cast<float*>(smem + L.off_h);
  float *vec_g = reinterpret_cast<float*>(smem + L.off_g), *vec_z = reinterpret_cast<float*>(smem + L.off_z);
  float *kv = reinterpret_cast<float*>(smem + L.off_kv), *gain_mlp = reinterpret_cast<float*>(smem + L.off_gain), *gain_kv = gain_mlp + p.d;
  float *fin = reinterpret_cast<float*>(smem + L.off_fin), *state = reinterpret_cast<float*>(smem + L.off_st);
  const T *s_wo = reinterpret_cast<const T*>(smem + L.off_wo), *s_wup = reinterpret_cast<const T*>(smem + L.off_wup),
          *s_wdn = reinterpret_cast<const T*>(smem + L.off_wdn), *s_wk = reinterpret_cast<const T*>(smem + L.off_wk), *s_wv = reinterpret_cast<const T*>(smem + L.off_wv);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)cluster_rank(), B = p.B, d = p.d, H = p.H, dff = p.dff, n = p.t1 - p.t0;
  const int b_lo = (int)(blockIdx.x / kCl) * NB, nb = B - b_lo < NB ? B - b_lo : NB;      // this cluster's sequences
  const int nd = d / kCl, nf = dff / kCl, d_lo = rank * nd, f_lo = rank * nf;
  const int pair = rank;                                       // (sequence, head) pair whose attention this CTA does
  const bool owner = pair < nb * H;
  SyncArea* const sync = p.sync;
  const bool dead = *reinterpret_cast<volatile unsigned*>(&sync->abort_flag) != 0;

  if (tid == 0) {
    *s_abort = dead ? 1 : 0;
    for (int i = 0; i < 6; ++i) mbar_init(bars + 8 * i, 1);
    mbar_init(bar_state, 2); mbar_init(bar_state + 8, 2);
    for (int i = 0; i < Handover::kReadyBars; ++i) mbar_init(bar_key + 8 * i, 1);
    for (int i = 0; i < kFin; ++i) mbar_init(bar_done + 8 * i, kFoldWarps);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(bar_c, (uint32_t)(nb * d * 4)); mbar_expect_tx(bar_h, (uint32_t)(nb * d * 4));
    mbar_expect_tx(bar_g, (uint32_t)(nb * dff * 4)); mbar_expect_tx(bar_z, (uint32_t)(nb * d * 4));
    mbar_expect_tx(bar_kv, 2 * kHeadDim * 4);
    // weight slices: contiguous rows, one bulk copy each
    const uint32_t wd = (uint32_t)((size_t)nd * d * sizeof(T)), wf = (uint32_t)((size_t)nf * d * sizeof(T));
    mbar_expect_tx(bar_w, 3 * wd + 2 * wf);
    auto in = [&](unsigned off, const void* W, size_t row, int K, uint32_t bytes) {
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   ::"r"(smem_u32(smem + off)), "l"(reinterpret_cast<const T*>(W) + row * K), "r"(bytes), "r"(bar_w) : "memory");
    };
    in(L.off_wo, p.w_o, d_lo, d, wd); in(L.off_wup, p.w_up, f_lo, d, wf); in(L.off_wdn, p.w_down, d_lo, dff, wf);
    in(L.off_wk, p.w_k, d_lo, d, wd); in(L.off_wv, p.w_v, d_lo, d, wd);
  }
  if (p.g_mlp) for (int k = tid; k < d; k += kSmThreads) gain_mlp[k] = to_f(reinterpret_cast<const T*>(p.g_mlp)[k]);
  if (p.g_kv) for (int k = tid; k < d; k += kSmThreads) gain_kv[k] = to_f(reinterpret_cast<const T*>(p.g_kv)[k]);
  __syncthreads();
  cluster_arrive_wait();                                       // every mbarrier exists before anyone sends

  const bool pre = (p.norm_flags & RT_NORM_PRE) != 0, qkn = (p.norm_flags & RT_NORM_QK) != 0;
  const bool kv_norm = pre && !(p.norm_flags & RT_NORM_SKIP_Z);
  const float inv_d = 1.0f / (float)d;

  if (warp >= kSmWarps) {
    // ------------------------------ attention: one (sequence, head) pair ------------------------------
    // One warp sits on the chain: it finishes query j + 1 with the pair of position j and publishes its value.  Four warps
    // hold the other queries of the leaf in registers (two lanes per query, 32 dimensions each), fold the pair into them while the
    // mat-vecs of the next step run, and leave the state of query j + 2 for the first warp.
    const int b = b_lo + pair / H, h = pair % H;
    const T* q = reinterpret_cast<const T*>(p.q);
    const float slope_l2 = p.alibi && owner ? p.alibi[h] * kLog2e : 0.f;
    const size_t row0 = (size_t)(p.t0 - p.row_off);
    if (owner && warp == kSmWarps) {
      T *kc = reinterpret_cast<T*>(p.k_cache), *vc = reinterpret_cast<T*>(p.v_cache);
      const float gk0 = qkn ? gain_at(reinterpret_cast<const T*>(p.g_k), h * kHeadDim + 2 * lane) : 1.f;
      const float gk1 = qkn ? gain_at(reinterpret_cast<const T*>(p.g_k), h * kHeadDim + 2 * lane + 1) : 1.f;
      // c goes to all CTAs: two dimensions per lane, one destination per instruction
      const uint32_t c_at = smem_u32(vec_c + (size_t)(b - b_lo) * d + h * kHeadDim + 2 * lane);
      auto publish = [&](float c0, float c1) {
        const float v[2] = {c0, c1};
#pragma unroll
        for (int r = 0; r < kCl; ++r) send(map_to(c_at, r), map_to(bar_c, r), v);
      };
      if (wait_bar(bar_state, 0, s_abort, sync)) {
        const float il = 1.f / state[kHeadDim + 1];
        const float2 o = *reinterpret_cast<const float2*>(state + 2 * lane);
        publish(o.x * il, o.y * il);
      }
      for (int j = 0; j < n; ++j) {
        float q0 = 0.f, q1 = 0.f;
        if (j + 1 < n) {
          const T* qp = q + ((row0 + j + 1) * B + b) * d + h * kHeadDim + 2 * lane;
          q0 = to_f(qp[0]); q1 = to_f(qp[1]);
          if (!wait_bar(bar_state + 8 * ((j + 1) & 1), ((j + 1) >> 1) & 1, s_abort, sync)) break;       // state of query j + 1
        }
        if (j >= kFin && !wait_bar(bar_done + 8 * Handover::slot(j), Handover::read_parity(j - kFin), s_abort, sync)) break;  // place of the pair j - 4
        if (!wait_bar(bar_kv, j & 1, s_abort, sync)) break;
        const float2 kr = *reinterpret_cast<const float2*>(kv + 2 * lane), vr = *reinterpret_cast<const float2*>(kv + kHeadDim + 2 * lane);
        const float rs = qkn ? rsqrtf(warp_sum(kr.x * kr.x + kr.y * kr.y) * (1.0f / kHeadDim) + p.eps) : 1.0f;
        const float k0 = round_T<T>(kr.x * rs * gk0), k1 = round_T<T>(kr.y * rs * gk1), v0 = round_T<T>(vr.x), v1 = round_T<T>(vr.y);
        if (j + 1 < n) {
          const float* st = state + ((j + 1) & 1) * kStateStride;
          const float s = warp_sum(q0 * k0 + q1 * k1) * p.scale_log2 - slope_l2;
          const float m_old = st[kHeadDim], m_new = fmaxf(m_old, s), corr = exp2f(m_old - m_new), pj = exp2f(s - m_new);
          const float il = 1.0f / (st[kHeadDim + 1] * corr + pj);
          const float2 o = *reinterpret_cast<const float2*>(st + 2 * lane);
          publish((o.x * corr + pj * v0) * il, (o.y * corr + pj * v1) * il);
        }
        float* f = fin + Handover::slot(j) * 2 * kHeadDim;
        *reinterpret_cast<float2*>(f + 2 * lane) = make_float2(k0, k1);
        *reinterpret_cast<float2*>(f + kHeadDim + 2 * lane) = make_float2(v0, v1);
        __syncwarp();
        if (lane == 0) {
          if (j + 1 < n) mbar_expect_tx(bar_kv, 2 * kHeadDim * 4);
          mbar_arrive(bar_key + 8 * Handover::ready_bar(j));
        }
        const size_t crow = ((size_t)(p.t0 + j) * B + b) * d + h * kHeadDim + 2 * lane;
        kc[crow] = from_f<T>(k0); kc[crow + 1] = from_f<T>(k1); vc[crow] = from_f<T>(v0); vc[crow + 1] = from_f<T>(v1);
      }
    } else if (owner) {
      const int ft = tid - (kSmWarps + 1) * 32, i = ft >> 1, e0 = (ft & 1) * 32;
      float qr[32], o[32], m = 0.f, l = 1.f;
      if (i < n) {
        const size_t row = (row0 + i) * B + b, at = row * d + h * kHeadDim + e0;
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
          float f[4];
          reinterpret_cast<const Vec4<T>*>(q + at + e)->to_float(f);
          const float4 ov = *reinterpret_cast<const float4*>(p.st_o + at + e);
          qr[e] = f[0]; qr[e + 1] = f[1]; qr[e + 2] = f[2]; qr[e + 3] = f[3];
          o[e] = ov.x; o[e + 1] = ov.y; o[e + 2] = ov.z; o[e + 3] = ov.w;
        }
        m = p.st_m[row * H + h]; l = p.st_l[row * H + h];
      } else {
#pragma unroll
        for (int e = 0; e < 32; ++e) { qr[e] = 0.f; o[e] = 0.f; }
      }
      auto leave_state = [&]() {                               // by the two lanes of one query
        float* st = state + (i & 1) * kStateStride;
#pragma unroll
        for (int e = 0; e < 32; e += 4) *reinterpret_cast<float4*>(st + e0 + e) = make_float4(o[e], o[e + 1], o[e + 2], o[e + 3]);
        if (e0 == 0) { st[kHeadDim] = m; st[kHeadDim + 1] = l; }
        mbar_arrive(bar_state + 8 * (i & 1));
      };
      if (i < 2 && i < n) leave_state();
      __syncwarp();
      for (int j = 0; j + 2 < n; ++j) {
        if (!wait_bar(bar_key + 8 * Handover::ready_bar(j), Handover::ready_parity(j), s_abort, sync)) break;
        const float* f = fin + Handover::slot(j) * 2 * kHeadDim;
        if ((ft | 31) >> 1 >= j + 2) {                         // some query of this warp is still open
          float s0 = 0.f, s1 = 0.f;
#pragma unroll
          for (int e = 0; e < 32; e += 4) {
            const float4 kk = *reinterpret_cast<const float4*>(f + e0 + e);
            s0 = fmaf(qr[e], kk.x, s0); s1 = fmaf(qr[e + 1], kk.y, s1); s0 = fmaf(qr[e + 2], kk.z, s0); s1 = fmaf(qr[e + 3], kk.w, s1);
          }
          float s = s0 + s1;
          s += __shfl_xor_sync(0xffffffffu, s, 1);
          s = s * p.scale_log2 - slope_l2 * (float)(i - j);
          const float m_new = fmaxf(m, s), corr = exp2f(m - m_new), pj = exp2f(s - m_new);
          m = m_new; l = l * corr + pj;
#pragma unroll
          for (int e = 0; e < 32; e += 4) {
            const float4 vv = *reinterpret_cast<const float4*>(f + kHeadDim + e0 + e);
            o[e] = fmaf(o[e], corr, pj * vv.x); o[e + 1] = fmaf(o[e + 1], corr, pj * vv.y);
            o[e + 2] = fmaf(o[e + 2], corr, pj * vv.z); o[e + 3] = fmaf(o[e + 3], corr, pj * vv.w);
          }
          if (i == j + 2) leave_state();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_done + 8 * Handover::slot(j));
      }
    }
  } else if (wait_bar(bar_w, 0, s_abort, sync)) {
    // ------------------------------ mat-vec warps ------------------------------
    constexpr int U = 2;                                       // rows per warp and round (W_up: 4)
    const T *x = reinterpret_cast<const T*>(p.x);
    T* z = reinterpret_cast<T*>(p.z);
    const int dest = lane & (kCl - 1);                         // lanes 0..15 send, one destination each
    float hown[NB][U];                                         // this warp's rows of h (nd <= 2 * 16 rows)
    const int r0 = warp * U;                                   // its rows of the d-wide matrices
    const bool has_d = r0 < nd;
    // per-phase times of the first CTA (profiling): phase ph's wait at 3 + 2 ph, its work at 2 + 2 ph
    const bool timing = TIMERS && blockIdx.x == 0 && tid == 0;
    unsigned long long t_mark = timing ? globaltimer_ns() : 0ull;
    auto stamp = [&](int at) {
      if (!timing) return;
      const unsigned long long now = globaltimer_ns();
      atomicAdd(&sync->phase_ns[at], now - t_mark);
      t_mark = now;
    };
    for (int j = 0; j < n; ++j) {
      const uint32_t par = j & 1;
      const bool more = tid == 0 && j + 1 < n;                 // this thread arms the barriers for the next step
      const size_t trow = (size_t)(p.t0 - p.row_off + j);
      float dummy[NB], y[U][NB];
      float xv[U][NB];
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int u = 0; u < U; ++u)
          xv[u][b] = has_d && b < nb ? to_f(x[(size_t)(b_lo + b) * p.x_bs + trow * p.x_ts + d_lo + r0 + u]) : 0.f;
      // h = x + alpha W_o c
      stamp(8);
      if (!wait_bar(bar_c, par, s_abort, sync)) break;
      stamp(3);
      if (more) mbar_expect_tx(bar_c, (uint32_t)(nb * d * 4));
      if (has_d) {
        rows_dot<T, U, NB, false>(s_wo + (size_t)r0 * d, vec_c, d, nullptr, lane, y, dummy);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          hown[b][0] = xv[0][b] + p.alpha * y[0][b]; hown[b][1] = xv[1][b] + p.alpha * y[1][b];
          if (b < nb && lane < kCl) send(map_to(smem_u32(vec_h + (size_t)b * d + d_lo + r0), dest), map_to(bar_h, dest), hown[b]);
        }
      }
      // g = GELU(W_up RMS(h))
      stamp(2);
      if (!wait_bar(bar_h, par, s_abort, sync)) break;
      stamp(5);
      if (more) mbar_expect_tx(bar_h, (uint32_t)(nb * d * 4));
      for (int f = warp * 4; f < nf; f += kSmWarps * 4) {
        float yg[4][NB], ss[NB];
        rows_dot<T, 4, NB, true>(s_wup + (size_t)f * d, vec_h, d, pre && p.g_mlp ? gain_mlp : nullptr, lane, yg, ss);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          const float rs = pre ? rsqrtf(ss[b] * inv_d + p.eps) : 1.0f;
          // every lane has all four sums; lane pairs would all compute the same GELU, so each lane of a quad takes one row
          const float mine = (lane & 3) == 0 ? yg[0][b] : (lane & 3) == 1 ? yg[1][b] : (lane & 3) == 2 ? yg[2][b] : yg[3][b];
          const float v = mine * rs, gl = 0.5f * v * (1.0f + erff(v * 0.70710678118654752f));
          float out[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) out[u] = __shfl_sync(0xffffffffu, gl, u);
          if (b < nb && lane < kCl) send(map_to(smem_u32(vec_g + (size_t)b * dff + f_lo + f), dest), map_to(bar_g, dest), out);
        }
      }
      // z = h + alpha W_down g
      stamp(4);
      if (!wait_bar(bar_g, par, s_abort, sync)) break;
      stamp(7);
      if (more) mbar_expect_tx(bar_g, (uint32_t)(nb * dff * 4));
      if (has_d) {
        rows_dot<T, U, NB, false>(s_wdn + (size_t)r0 * dff, vec_g, dff, nullptr, lane, y, dummy);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          const float zv[2] = {round_T<T>(hown[b][0] + p.alpha * y[0][b]), round_T<T>(hown[b][1] + p.alpha * y[1][b])};
          if (b >= nb) continue;
          if (lane < kCl) send(map_to(smem_u32(vec_z + (size_t)b * d + d_lo + r0), dest), map_to(bar_z, dest), zv);
          if (lane < U) z[(size_t)(b_lo + b) * p.z_bs + trow * p.z_ts + d_lo + r0 + lane] = from_f<T>(lane ? zv[1] : zv[0]);
        }
      }
      // raw k, v from RMS(z), to the CTA that owns the head
      stamp(6);
      if (!wait_bar(bar_z, par, s_abort, sync)) break;
      stamp(9);
      if (more) mbar_expect_tx(bar_z, (uint32_t)(nb * d * 4));
      for (int r = warp * U; r < 2 * nd; r += kSmWarps * U) {
        const bool second = r >= nd;
        const int rl = second ? r - nd : r, col = d_lo + rl;
        float ss[NB];
        rows_dot<T, U, NB, true>((second ? s_wv : s_wk) + (size_t)rl * d, vec_z, d, kv_norm && p.g_kv ? gain_kv : nullptr, lane, y, ss);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          const float rs = kv_norm ? rsqrtf(ss[b] * inv_d + p.eps) : 1.0f;
          const float v[2] = {y[0][b] * rs, y[1][b] * rs};
          const int to = b * H + col / kHeadDim;               // the pair's CTA
          if (b < nb && lane == 0) send(map_to(smem_u32(kv + (second ? kHeadDim : 0) + col % kHeadDim), to), map_to(bar_kv, to), v);
        }
      }
    }
  }
  // nobody leaves while a store to its shared memory can still be on its way
  __syncwarp();
  cluster_arrive_wait();
}

}  // namespace

// Clusters of 16 that run at the same time (measured: with eight, the last one waits for the others).
constexpr int kClusters = 7;

// Whether the shape runs on this kernel with leaves of `leaf` positions (pure arithmetic), and how many sequences a cluster
// carries: one to three, whatever makes rounds of clusters x time per round least (a step with 2 or 3 sequences measured about 1.35 and
// 1.7 times one with a single sequence at d = 128 .. 256; that one 3.1, 3.3, 4.0, 4.5, 5.8 and 6.3 us at d = 64, 128, ... 384 in bf16).
//
// The values between the phases stay fp32 here, so fp32 layers always stay (the generic kernel takes three times as long or more), and bf16
// layers up to the time that the same batch takes with its values in bf16 as slices of 16 sequences one after the other through the tensor-core leaf
// kernel, 11.3 us each, or, above 48, as dense products, 38 us.  Per 256 positions at d = 384: 15 sequences take 4.3 ms here (two rounds) and 2.9
// there, 32 6.8 and 6.0, 64 11.4 and 9.8, but 24 4.6 and 5.9; up to d = 320 every batch is within the bound.  (The group kernel, also on
// bf16 values, is the fastest from about two rounds on: 3.8 ms against 5.9 for d = 256, B = 48; it takes what is beyond the bound.)
bool leaf_small_shape(int dtype, int B, int d, int H, int dff, int leaf, size_t max_smem, LeafSmallLaunch* out) {
  if (d % 64 || dff % 64 || d > 512 || leaf > kSmLeafMax) return false;
  int nb = 0;
  float best = 0.f;
  for (int k = 1; k <= 3 && k * H <= kCl; ++k) {
    const float cost = ceil_div(ceil_div(B, k), kClusters) * (0.65f + 0.35f * k);
    if (!nb || cost < best) { nb = k; best = cost; }
  }
  if (!nb) return false;
  const size_t es = dtype == RT_BF16 ? 2 : 4;
  const SmallLayout L = small_layout(es, nb, d, dff);
  if (L.total > max_smem) return false;
  const float weights_kb = (float)(L.total - L.off_wo) * (1.0f / 1024.0f);
  out->nb = nb; out->leaf = leaf; out->smem = L.total; out->step_us = best * (3.0f + weights_kb * (1.0f / 60.0f));
  return dtype != RT_BF16 || out->step_us <= (B > 48 ? 38.0f : 11.3f * ceil_div(B, 16));
}

cudaError_t leaf_small_launch(int dtype, const LeafParams& p, const LeafSmallLaunch& l, cudaStream_t s) {
  const SmallLayout L = small_layout(dtype == RT_BF16 ? 2 : 4, l.nb, p.d, p.dff);
  auto go = [&](auto kernel) -> cudaError_t {
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), (int)L.total);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kCl * ceil_div(p.B, l.nb)); cfg.blockDim = dim3(kSmThreads); cfg.dynamicSmemBytes = L.total; cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kCl; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, p, L);
  };
  auto pick = [&](auto t, auto nb) -> cudaError_t {
    using T = decltype(t);
    constexpr int NB = decltype(nb)::value;
    return p.timers ? go(leaf_small_kernel<T, NB, true>) : go(leaf_small_kernel<T, NB, false>);
  };
  auto by_nb = [&](auto t) -> cudaError_t {
    if (l.nb == 1) return pick(t, std::integral_constant<int, 1>{});
    if (l.nb == 2) return pick(t, std::integral_constant<int, 2>{});
    return pick(t, std::integral_constant<int, 3>{});
  };
  return dtype == RT_BF16 ? by_nb(__nv_bfloat16{}) : by_nb(0.f);
}

}  // namespace rt
