// The reverse loop of the backward pass over one leaf, bf16 weights, up to eight sequences per launch (rt_backward.cu states
// the recurrence): persistent CTAs with tensor-core mat-vecs and exchange words, the mirror image of rt_leaf_mma.cu.
//
// Per position i (descending) a chain of five exchanges:
//   dk_raw_i | dv_i -> dr_i = dk_raw W_k + dv W_v -> Gz = dz + RMS backward(dr), dpre = (alpha Gz W_down) GELU' -> du = dpre W_up
//   -> dh = Gz + RMS backward(du), dc = alpha dh W_o -> the query's share of d(k_j, v_j), j < i; then dk_raw_{i-1} | dv_{i-1}
//   * every exchanged value is an entry of an array that stage 3 needs anyway ([position, sequence, ...] fp32), written once.  The
//     arrays are filled with 0xFFFFFFFF (a NaN that no arithmetic produces) before the loop, so the entries are their own flags and a
//     consumer polls them directly: no barrier across CTAs, no second round trip.  (Five grid barriers per position took 30 us.)
//   * products run as bf16 m16n8k16 MMAs on the exact split x = hi + mid + lo of every fp32 value into three bf16 terms (24 bits), which
//     take the MMA's 16 rows: up to four sequences all three terms of each (one MMA per 16 x 8 block of weights), up to eight hi and mid, lo in a
//     second one.  So nothing is lost against fp32 fused multiply-adds with the bf16 weights.  (tf32 MMAs with two 11-bit terms took 65
//     cycles each, eight times a bf16 one: 20 us per position.)  K split over eight warps, weights (transposed once per call) resident in
//     shared memory for the leaf.
//   * five attention warps per (sequence, head): one on the chain (finishes the pair of position i-1 with the query of position i and
//     publishes it), four that hold d(k, v) of the leaf's 64 positions in registers (two lanes per position) and absorb the query
//     while the products run.
#include <cuda_bf16.h>
#include <string.h>

#include "rt_handover.h"
#include "rt_kernels.h"
#include "rt_tc.cuh"

namespace rt {

namespace {

constexpr int kBMma = 8, kBFold = 4;
constexpr int kBFold0 = kBMma, kBChain = kBMma + kBFold;     // warps: products, fold, chain, three idle ones (whole warpgroups for setmaxnreg)
constexpr int kBThreads = 512;
constexpr int kBRegsMma = 160, kBRegsAtt = 96;               // (160 + 96) * 256 = 65536
constexpr int kBMmaThreads = kBMma * 32;
constexpr int kBLeaf = 64;
constexpr int kBRing = Handover::kSlots;          // queries handed to the fold warps
constexpr int kKvRow = 144;                       // floats of one position's k | v in shared memory: halves 36 apart (no bank conflicts)
constexpr unsigned kBEmpty = 0xffffffffu;

struct BLoopLayout {
  int max_nd, max_nf, nt_d, nt_f, stride_2d, stride_d, stride_f;
  uint32_t off_red, off_ssq, off_kv, off_state, off_ring, off_pair, off_dn, off_up, off_o, total;
};
BLoopLayout bloop_layout(int d, int dff, int grid) {
  BLoopLayout L;
  L.max_nd = 2 * ceil_div(d / 2, grid); L.max_nf = 2 * ceil_div(dff / 2, grid);
  L.nt_d = ceil_div(L.max_nd, 8); L.nt_f = ceil_div(L.max_nf, 8);
  L.stride_2d = 2 * d + 16; L.stride_d = d + 16; L.stride_f = dff + 16;      // 8-byte fragment loads of 8 rows without conflicts
  uint32_t o = 256;
  auto take = [&](size_t n) { o = (o + 127) / 128 * 128; const uint32_t at = o; o += (uint32_t)n; return at; };
  const int tiles = L.nt_f > L.nt_d ? L.nt_f : L.nt_d;
  L.off_red = take((size_t)2 * tiles * kBMma * 32 * 8);
  L.off_ssq = take((size_t)2 * kBMma * 8 * 8);
  L.off_kv = take((size_t)kBLeaf * kKvRow * 4);
  L.off_state = take((size_t)2 * 2 * kHeadDim * 4);
  L.off_ring = take((size_t)kBRing * (2 * kHeadDim + 4) * 4);
  L.off_pair = take((size_t)L.max_nd * L.stride_2d * 2);
  L.off_dn = take((size_t)L.max_nf * L.stride_d * 2);
  L.off_up = take((size_t)L.max_nd * L.stride_f * 2);
  L.off_o = take((size_t)L.max_nd * L.stride_d * 2);
  L.total = o;
  return L;
}

__device__ __forceinline__ float blo(unsigned u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bhi(unsigned u) { return __uint_as_float(u & 0xffff0000u); }
__device__ __forceinline__ uint4 bl_ld4_if(const void* p, unsigned on) {
  unsigned long long a = 0ull, b = 0ull;
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %3, 0;\n @q ld.relaxed.gpu.global.v2.u64 {%0,%1}, [%2];\n}"
               : "+l"(a), "+l"(b) : "l"(p), "r"(on) : "memory");
  return make_uint4((unsigned)a, (unsigned)(a >> 32), (unsigned)b, (unsigned)(b >> 32));
}
__device__ __forceinline__ uint2 bl_ld2(const void* p) {
  unsigned long long a;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(a) : "l"(p) : "memory");
  return make_uint2((unsigned)a, (unsigned)(a >> 32));
}
__device__ __forceinline__ void bl_st2(void* p, float a, float b) {
  const unsigned long long w = ((unsigned long long)__float_as_uint(b) << 32) | __float_as_uint(a);
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ void bl_mma(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// A pair of fp32 values as three pairs of bf16 whose sums are the values.
__device__ __forceinline__ void split3(float x0, float x1, unsigned& hi, unsigned& mid, unsigned& lo) {
  auto pk = [](float a, float b) { const __nv_bfloat162 v = __floats2bfloat162_rn(a, b); return *reinterpret_cast<const unsigned*>(&v); };
  hi = pk(x0, x1);
  x0 -= blo(hi); x1 -= bhi(hi);
  mid = pk(x0, x1);
  lo = pk(x0 - blo(mid), x1 - bhi(mid));
}
__device__ __forceinline__ float gelu_grad(float a) {          // d/da [a Phi(a)] = Phi(a) + a phi(a)
  return 0.5f * (1.f + erff(a * 0.70710678118654752f)) + a * 0.3989422804014327f * __expf(-0.5f * a * a);
}
__device__ __forceinline__ void b_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kBMmaThreads) : "memory"); }
__device__ __noinline__ bool bl_give_up(SyncArea* s, volatile int* s_abort, unsigned long long* t_start) {
  if (*s_abort) return true;
  if (*reinterpret_cast<volatile unsigned*>(&s->abort_flag)) { *s_abort = 1; return true; }
  const unsigned long long now = globaltimer_ns();
  if (*t_start == 0) { *t_start = now; return false; }
  if (now - *t_start <= kWaitLimitNs) return false;
  s->status = RT_ERR_TIMEOUT;
  __threadfence();
  atomicExch(&s->abort_flag, 1u);
  *s_abort = 1;
  return true;
}
// Whole warp; after a wait that ran out everybody goes on to the end (barriers need every warp).
__device__ __forceinline__ void bl_wait(uint32_t bar, uint32_t parity, SyncArea* s, volatile int* s_abort) {
  unsigned spins = 0;
  unsigned long long t0 = 0;
  while (!mbar_try_wait(bar, parity))
    if ((++spins & 255u) == 0u && bl_give_up(s, s_abort, &t0)) break;
  __syncwarp();
}
__device__ __forceinline__ uint2 bl_poll2(const void* p, SyncArea* s, volatile int* s_abort) {
  unsigned spins = 0;
  unsigned long long t0 = 0;
  uint2 w;
  while (true) {
    w = bl_ld2(p);
    if (__all_sync(0xffffffffu, w.x != kBEmpty && w.y != kBEmpty)) break;
    if ((++spins & 63u) == 0u && __any_sync(0xffffffffu, bl_give_up(s, s_abort, &t0))) break;
  }
  return w;
}

// SMALL: at most four sequences (all three terms of each in one MMA).
template <bool SMALL>
__global__ void __launch_bounds__(kBThreads, 1) bwd_leaf_kernel(const __grid_constant__ BwdLeafParams p, const BLoopLayout L) {
  extern __shared__ __align__(128) unsigned char smem[];
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem);
  const uint32_t bars = smem_u32(smem + 16);
  // weights; state of the pair that is finished next (even, odd); query handed over, absorbed (ring, rt_handover.h)
  const uint32_t w_bar = bars, bar_state = bars + 8, bar_key = bars + 24, bar_done = bar_key + 8 * Handover::kReadyBars;
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int G = gridDim.x, cta = blockIdx.x, B = p.B, d = p.d, H = p.H, dff = p.dff;
  const int d_lo = 2 * (int)((long long)(d / 2) * cta / G), nd = 2 * (int)((long long)(d / 2) * (cta + 1) / G) - d_lo;
  const int f_lo = 2 * (int)((long long)(dff / 2) * cta / G), nf = 2 * (int)((long long)(dff / 2) * (cta + 1) / G) - f_lo;
  SyncArea* const sync = p.sync;
  const bool owner = cta < B * H;

  if (tid == 0) {
    *s_abort = *reinterpret_cast<volatile unsigned*>(&sync->abort_flag) ? 1 : 0;
    mbar_init(w_bar, 1); mbar_init(bar_state, 2); mbar_init(bar_state + 8, 2);
    for (int i = 0; i < Handover::kReadyBars; ++i) mbar_init(bar_key + 8 * i, 1);
    for (int i = 0; i < kBRing; ++i) mbar_init(bar_done + 8 * i, kBFold);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(w_bar, (uint32_t)(((size_t)3 * nd * d + (size_t)nf * d + (size_t)nd * dff) * 2));
  }
  __syncthreads();

  if (warp >= kBMma) {
    // ------------------------------ attention: one (sequence, head) pair ------------------------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kBRegsAtt));
    if (warp == kBChain + 1 && cta >= G - 4) {
      // Rows that nobody has touched since the sweep (W_up u, h, dz, z) would each cost a trip to HBM in the middle of a step: an idle
      // warp of four CTAs asks L2 for them, one array each, two positions ahead of the chain (whose first output it watches).
      const int which = G - 1 - cta, width = which == 0 ? dff : d, esz = which == 3 ? 2 : 4;
      for (int i = p.e0 + 1; i >= p.s0; --i) {
        if (i < p.e0 - 2) {
          unsigned spins = 0;
          unsigned long long t0 = 0;
          while (bl_ld2(p.dr + ((size_t)(i + 2) * p.Bs + p.b0) * d).x == kBEmpty) {
            __nanosleep(200);
            if ((++spins & 63u) == 0u && bl_give_up(sync, s_abort, &t0)) return;
          }
        }
        if (i >= p.e0) continue;
        for (int bb = 0; bb < B; ++bb) {
          const size_t seq = (size_t)(p.b0 + bb), row = (size_t)i * p.Bs + seq;
          const unsigned char* a = which == 0 ? reinterpret_cast<const unsigned char*>(p.act + row * dff) : which == 1 ? reinterpret_cast<const unsigned char*>(p.h + row * d)
                                 : which == 2 ? reinterpret_cast<const unsigned char*>(p.dz + seq * p.dz_bs + (size_t)i * p.dz_ts)
                                              : reinterpret_cast<const unsigned char*>(reinterpret_cast<const __nv_bfloat16*>(p.z) + seq * p.z_bs + (size_t)i * p.z_ts);
          for (int e = lane * 128; e < width * esz; e += 32 * 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(a + e));
        }
      }
      return;
    }
    if (!owner || warp > kBChain) return;
    const int b = cta / H, h = cta % H;
    const size_t rstride = (size_t)p.Bs * d, col = (size_t)(p.b0 + b) * d + h * kHeadDim;      // a position's row; this pair's columns
    const size_t sstride = (size_t)p.Bs * H, scol = (size_t)(p.b0 + b) * H + h;
    const float slope = p.alibi ? p.alibi[h] * kLog2e : 0.f;
    float* kv = reinterpret_cast<float*>(smem + L.off_kv);
    float* state = reinterpret_cast<float*>(smem + L.off_state);                               // [2][dk 64 | dv 64]
    float* ring = reinterpret_cast<float*>(smem + L.off_ring);                                 // [4][q 64 | dc 64 | lse, D]
    constexpr int kRingRow = 2 * kHeadDim + 4;
    if (warp < kBChain) {
      // four warps: positions of the leaf, two lanes each (32 dimensions)
      const int ft = tid - kBFold0 * 32, jj = ft >> 1, e0 = (ft & 1) * 32, j = p.s0 + jj;
      float dk[32], dv[32];
      float* kr = kv + jj * kKvRow + (ft & 1) * 36;
      float* vr = kr + 72;
      if (j < p.e0) {
        const size_t at = (size_t)j * rstride + col + e0;
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
          *reinterpret_cast<float4*>(kr + e) = *reinterpret_cast<const float4*>(p.k + at + e);
          *reinterpret_cast<float4*>(vr + e) = *reinterpret_cast<const float4*>(p.v + at + e);
          const float4 a = *reinterpret_cast<const float4*>(p.dK + at + e), c = *reinterpret_cast<const float4*>(p.dV + at + e);
          dk[e] = a.x; dk[e + 1] = a.y; dk[e + 2] = a.z; dk[e + 3] = a.w;
          dv[e] = c.x; dv[e + 1] = c.y; dv[e + 2] = c.z; dv[e + 3] = c.w;
        }
      } else {
#pragma unroll
        for (int e = 0; e < 32; ++e) { dk[e] = 0.f; dv[e] = 0.f; }
        for (int e = 0; e < 32; ++e) { kr[e] = 0.f; vr[e] = 0.f; }
      }
      auto leave_state = [&]() {                               // by the two lanes of one position
        const int idx = p.e0 - 1 - j;
        float* st = state + (idx & 1) * 2 * kHeadDim + e0;
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
          *reinterpret_cast<float4*>(st + e) = make_float4(dk[e], dk[e + 1], dk[e + 2], dk[e + 3]);
          *reinterpret_cast<float4*>(st + kHeadDim + e) = make_float4(dv[e], dv[e + 1], dv[e + 2], dv[e + 3]);
        }
        mbar_arrive(bar_state + 8 * (idx & 1));
      };
      if (j < p.e0 && j >= p.e0 - 2) leave_state();
      __syncwarp();
      int step = 0;
      for (int i = p.e0 - 1; i >= p.s0 + 2; --i, ++step) {
        bl_wait(bar_key + 8 * Handover::ready_bar(step), Handover::ready_parity(step), sync, s_abort);
        const float* f = ring + Handover::slot(step) * kRingRow;
        if (p.s0 + (ft & ~31) / 2 <= i - 2) {                  // some position of this warp is still open
          float s0 = 0.f, s1 = 0.f, t0 = 0.f, t1 = 0.f;
#pragma unroll 2
          for (int e = 0; e < 32; e += 4) {
            const float4 kk = *reinterpret_cast<const float4*>(kr + e), vv = *reinterpret_cast<const float4*>(vr + e);
            const float4 qq = *reinterpret_cast<const float4*>(f + e0 + e), cc = *reinterpret_cast<const float4*>(f + kHeadDim + e0 + e);
            s0 = fmaf(qq.x, kk.x, s0); s1 = fmaf(qq.y, kk.y, s1); s0 = fmaf(qq.z, kk.z, s0); s1 = fmaf(qq.w, kk.w, s1);
            t0 = fmaf(cc.x, vv.x, t0); t1 = fmaf(cc.y, vv.y, t1); t0 = fmaf(cc.z, vv.z, t0); t1 = fmaf(cc.w, vv.w, t1);
          }
          float s = s0 + s1, dp = t0 + t1;
          s += __shfl_xor_sync(0xffffffffu, s, 1);
          dp += __shfl_xor_sync(0xffffffffu, dp, 1);
          if (j <= i - 2) {
            const float pr = exp2f(s * p.scale_log2 - slope * (float)(i - j) - f[2 * kHeadDim]);
            const float ds = pr * (dp - f[2 * kHeadDim + 1]) * p.scale;
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
              const float4 qq = *reinterpret_cast<const float4*>(f + e0 + e), cc = *reinterpret_cast<const float4*>(f + kHeadDim + e0 + e);
              dk[e] = fmaf(ds, qq.x, dk[e]); dk[e + 1] = fmaf(ds, qq.y, dk[e + 1]); dk[e + 2] = fmaf(ds, qq.z, dk[e + 2]); dk[e + 3] = fmaf(ds, qq.w, dk[e + 3]);
              dv[e] = fmaf(pr, cc.x, dv[e]); dv[e + 1] = fmaf(pr, cc.y, dv[e + 1]); dv[e + 2] = fmaf(pr, cc.z, dv[e + 2]); dv[e + 3] = fmaf(pr, cc.w, dv[e + 3]);
            }
            if (j == i - 2) leave_state();
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_done + 8 * Handover::slot(step));
      }
      return;
    }
    // the warp on the chain: two dimensions per lane
    const int e2 = 2 * lane;
    const __nv_bfloat16* g_k = reinterpret_cast<const __nv_bfloat16*>(p.g_k);
    const float g0 = p.qk ? gain_at(g_k, h * kHeadDim + e2) : 1.f, g1 = p.qk ? gain_at(g_k, h * kHeadDim + e2 + 1) : 1.f;
    auto f2 = [&](const float* a, int i) { return *reinterpret_cast<const float2*>(a + (size_t)i * rstride + col + e2); };
    // qkRMS backward of dk through k = qkRMS(kraw) and everything out
    auto publish = [&](int j, float dk0, float dk1, float dv0, float dv1, float2 u, float inv) {
      const size_t at = (size_t)j * rstride + col + e2;
      float r0 = dk0, r1 = dk1;
      if (p.qk) {
        const float t0 = dk0 * g0, t1 = dk1 * g1, mean = warp_sum(t0 * u.x + t1 * u.y) * inv * (1.0f / kHeadDim);
        r0 = inv * (t0 - u.x * inv * mean); r1 = inv * (t1 - u.y * inv * mean);
      }
      bl_st2(p.dkraw + at, r0, r1);
      bl_st2(p.dvf + at, dv0, dv1);
      *reinterpret_cast<float2*>(p.dK + at) = make_float2(dk0, dk1);
    };
    auto inv_of = [&](float2 u) { return rsqrtf(warp_sum(u.x * u.x + u.y * u.y) * (1.0f / kHeadDim) + p.eps); };
    {
      const float2 u = f2(p.kraw, p.e0 - 1);
      const float inv = inv_of(u);
      bl_wait(bar_state, 0, sync, s_abort);
      const float2 a = *reinterpret_cast<const float2*>(state + e2), c = *reinterpret_cast<const float2*>(state + kHeadDim + e2);
      publish(p.e0 - 1, a.x, a.y, c.x, c.y, u, inv);
    }
    int step = 0;
    for (int i = p.e0 - 1; i >= p.s0; --i, ++step) {
      const bool more = i > p.s0;
      const float2 q = f2(p.q, i), cv = f2(p.c, i), kt = f2(p.kt, i), vt = f2(p.vt, i);
      const float lse = p.lse[(size_t)i * sstride + scol];
      float2 k1 = make_float2(0.f, 0.f), v1 = k1, u = k1;
      if (more) { k1 = f2(p.k, i - 1); v1 = f2(p.v, i - 1); u = f2(p.kraw, i - 1); }
      const float pt = exp2f(warp_sum(q.x * kt.x + q.y * kt.y) * p.scale_log2 - lse);
      const float pr = exp2f(warp_sum(q.x * k1.x + q.y * k1.y) * p.scale_log2 - slope - lse);
      const float inv = inv_of(u);
      if (more) bl_wait(bar_state + 8 * ((step + 1) & 1), ((step + 1) >> 1) & 1, sync, s_abort);          // state of position i - 1
      const float* st = state + ((step + 1) & 1) * 2 * kHeadDim;
      const float2 sk = *reinterpret_cast<const float2*>(st + e2), sv = *reinterpret_cast<const float2*>(st + kHeadDim + e2);
      const uint2 w = bl_poll2(p.dc + (size_t)i * rstride + col + e2, sync, s_abort);
      const float c0 = __uint_as_float(w.x), c1 = __uint_as_float(w.y);
      const float D = warp_sum(c0 * cv.x + c1 * cv.y), dp = warp_sum(c0 * v1.x + c1 * v1.y);
      if (more) {
        const float ds = pr * (dp - D) * p.scale;
        publish(i - 1, fmaf(ds, q.x, sk.x), fmaf(ds, q.y, sk.y), fmaf(pr, c0, sv.x), fmaf(pr, c1, sv.y), u, inv);
      }
      // off the chain: hand the query to the fold warps, then the temporary pair
      if (i >= p.s0 + 2) {
        if (step >= kBRing) bl_wait(bar_done + 8 * Handover::slot(step), Handover::read_parity(step - kBRing), sync, s_abort);
        float* f = ring + Handover::slot(step) * kRingRow;
        *reinterpret_cast<float2*>(f + e2) = q;
        *reinterpret_cast<float2*>(f + kHeadDim + e2) = make_float2(c0, c1);
        if (lane == 0) { f[2 * kHeadDim] = lse; f[2 * kHeadDim + 1] = D; }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_key + 8 * Handover::ready_bar(step));
      }
      const float dst = pt * (warp_sum(c0 * vt.x + c1 * vt.y) - D) * p.scale;
      const size_t at = (size_t)i * rstride + col + e2;
      *reinterpret_cast<float2*>(p.dkt + at) = make_float2(dst * q.x, dst * q.y);
      *reinterpret_cast<float2*>(p.dvt + at) = make_float2(pt * c0, pt * c1);
      if (lane == 0) p.D[(size_t)i * sstride + scol] = D;
    }
    return;
  }

  // ------------------------------ products ------------------------------
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kBRegsMma));
  if (warp == 0) {
    // the CTA's rows of the transposed weights, one bulk copy each
    auto stage = [&](uint32_t off, int stride, const void* W, int row_lo, int rows, int K, int at) {
      for (int r = lane; r < rows; r += 32)
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem_u32(smem + off) + (uint32_t)((r * stride + at) * 2)), "l"(reinterpret_cast<const __nv_bfloat16*>(W) + (size_t)(row_lo + r) * K),
                       "r"((uint32_t)K * 2u), "r"(w_bar) : "memory");
    };
    stage(L.off_pair, L.stride_2d, p.wkT, d_lo, nd, d, 0);
    stage(L.off_pair, L.stride_2d, p.wvT, d_lo, nd, d, d);
    stage(L.off_dn, L.stride_d, p.wdnT, f_lo, nf, d, 0);
    stage(L.off_up, L.stride_f, p.wupT, d_lo, nd, dff, 0);
    stage(L.off_o, L.stride_d, p.woT, d_lo, nd, d, 0);
  }
  constexpr int KC = 8;                                        // k-steps of 16 per round
  const int g = lane >> 2, c = lane & 3, sq = SMALL ? g & 3 : g;  // sq: sequence of this lane's rows
  const bool has = sq < B;
  const size_t brow = (size_t)(p.b0 + (has ? sq : 0));
  const float inv_d = 1.0f / (float)d;
  const __nv_bfloat16 *z = reinterpret_cast<const __nv_bfloat16*>(p.z), *g_kv = reinterpret_cast<const __nv_bfloat16*>(p.g_kv), *g_mlp = reinterpret_cast<const __nv_bfloat16*>(p.g_mlp);
  float gz[KC][4];                                             // Gz of this warp's stretch of d
  int buf = 0;
  bl_wait(w_bar, 0, sync, s_abort);

  for (int i = p.e0 - 1; i >= p.s0; --i) {
    const size_t row = (size_t)i * p.Bs + brow;
#pragma unroll 1
    for (int ph = 0; ph < 4; ++ph) {                           // 0: W_k | W_v   1: W_down   2: W_up   3: W_o
      const int K = ph == 0 ? 2 * d : ph == 2 ? dff : d, stride = ph == 0 ? L.stride_2d : ph == 2 ? L.stride_f : L.stride_d;
      const int rows = ph == 1 ? nf : nd, tiles = ph == 1 ? L.nt_f : L.nt_d;
      const bool norm = ph == 1 ? p.z_norm != 0 : p.pre != 0;
      const unsigned char* wbase = smem + (ph == 0 ? L.off_pair : ph == 1 ? L.off_dn : ph == 2 ? L.off_up : L.off_o);
      const int n_ks = K / 16, per = (n_ks + kBMma - 1) / kBMma, ks0 = warp * per, ks1 = ks0 + per < n_ks ? ks0 + per : n_ks;
      const int kb = ks0 * 16 + 4 * c;                         // this lane's first k
      float acc0[4] = {0.f, 0.f, 0.f, 0.f}, acc1[4] = {0.f, 0.f, 0.f, 0.f};
      float2* red = reinterpret_cast<float2*>(smem + L.off_red) + (size_t)buf * (L.nt_f > L.nt_d ? L.nt_f : L.nt_d) * kBMma * 32;
      buf ^= 1;
      if (ks0 >= ks1)
        for (int t = 0; t < tiles; ++t) red[(t * kBMma + warp) * 32 + lane] = make_float2(0.f, 0.f);
      // this warp's stretch of the polled vector (phase 0: the first four warps dk_raw, the others dv)
      const float* src = ph == 0 ? (warp < kBMma / 2 ? p.dkraw + row * d + kb : p.dvf + row * d + (kb - d)) : ph == 1 ? p.dr + row * d + kb : ph == 2 ? p.dpre + row * dff + kb : p.du + row * d + kb;
      auto load = [&](uint4 (&v)[KC], int s0) {
#pragma unroll
        for (int s = 0; s < KC; ++s) { const bool on = has && ks0 + s0 + s < ks1; v[s] = bl_ld4_if(src + 16 * (s0 + s), on ? 1u : 0u); }
      };
      uint4 xv[KC], xn[KC];                                    // this round's values; the next round's, or (norm phases, one round) u
      if (ph & 1) {
        // what the norm backward needs besides the polled vector, fetched before the wait: u in xn, the term added in gz
#pragma unroll
        for (int s = 0; s < KC; ++s) {
          const int k = ks0 + s < ks1 ? kb + 16 * s : 4 * c;
          if (ph == 1) {
            const float4 a = *reinterpret_cast<const float4*>(p.dz + brow * p.dz_bs + (size_t)i * p.dz_ts + k);
            gz[s][0] = a.x; gz[s][1] = a.y; gz[s][2] = a.z; gz[s][3] = a.w;
            const uint2 w = *reinterpret_cast<const uint2*>(z + brow * p.z_bs + (size_t)i * p.z_ts + k);
            xn[s] = make_uint4(w.x << 16, w.x & 0xffff0000u, w.y << 16, w.y & 0xffff0000u);
          } else xn[s] = *reinterpret_cast<const uint4*>(p.h + row * d + k);
        }
      }
      load(xv, 0);
#pragma unroll 1
      for (int s0 = 0; ks0 + s0 < ks1; s0 += KC) {
        if (ks0 + s0 + KC < ks1) load(xn, s0 + KC);
        unsigned spins = 0;
        unsigned long long t0 = 0;
        while (true) {                                         // a word that is not there yet is the largest there is
          unsigned m = 0;
#pragma unroll
          for (int s = 0; s < KC; ++s) m = max(max(m, max(xv[s].x, xv[s].y)), max(xv[s].z, xv[s].w));
          if (__all_sync(0xffffffffu, m != kBEmpty)) break;
          if ((++spins & 63u) == 0u && __any_sync(0xffffffffu, bl_give_up(sync, s_abort, &t0))) break;
          load(xv, s0);
        }
        float x[KC][4], uu[KC][4];
#pragma unroll
        for (int s = 0; s < KC; ++s) {
          x[s][0] = __uint_as_float(xv[s].x); x[s][1] = __uint_as_float(xv[s].y); x[s][2] = __uint_as_float(xv[s].z); x[s][3] = __uint_as_float(xv[s].w);
          uu[s][0] = __uint_as_float(xn[s].x); uu[s][1] = __uint_as_float(xn[s].y); uu[s][2] = __uint_as_float(xn[s].z); uu[s][3] = __uint_as_float(xn[s].w);
        }
        if (ph & 1) {
          // Gz = dz + RMS backward of dr through RMS(z);  dh = Gz + RMS backward of du through RMS(h)
          float inv = 0.f, coef = 0.f;
          if (norm) {
            const __nv_bfloat16* gain = ph == 1 ? g_kv : g_mlp;
            float ss = 0.f, tu = 0.f;
#pragma unroll
            for (int s = 0; s < KC; ++s) {                     // (steps beyond the stretch: x = 0, u masked)
              const int k = ks0 + s < ks1 ? kb + 16 * s : 4 * c;
              const float on = ks0 + s < ks1 ? 1.f : 0.f;
              if (gain) {
                const uint2 w = *reinterpret_cast<const uint2*>(gain + k);
                x[s][0] *= blo(w.x); x[s][1] *= bhi(w.x); x[s][2] *= blo(w.y); x[s][3] *= bhi(w.y);
              }
#pragma unroll
              for (int e = 0; e < 4; ++e) { ss = fmaf(on * uu[s][e], uu[s][e], ss); tu = fmaf(x[s][e], uu[s][e], tu); }
            }
            ss += __shfl_xor_sync(0xffffffffu, ss, 1); ss += __shfl_xor_sync(0xffffffffu, ss, 2);
            tu += __shfl_xor_sync(0xffffffffu, tu, 1); tu += __shfl_xor_sync(0xffffffffu, tu, 2);
            float2* sums = reinterpret_cast<float2*>(smem + L.off_ssq) + (ph >> 1) * kBMma * 8;
            if (c == 0) sums[warp * 8 + g] = make_float2(ss, tu);
            b_sync();
            ss = 0.f; tu = 0.f;
#pragma unroll
            for (int w = 0; w < kBMma; ++w) { const float2 v = sums[w * 8 + g]; ss += v.x; tu += v.y; }
            inv = rsqrtf(ss * inv_d + p.eps);
            coef = tu * inv * inv_d * inv;                     // mean(t uh) inv:  du = inv t - u inv (inv mean)
          } else inv = 1.f;
#pragma unroll
          for (int s = 0; s < KC; ++s) {
#pragma unroll
            for (int e = 0; e < 4; ++e) x[s][e] = gz[s][e] + inv * (x[s][e] - (norm ? uu[s][e] * coef : 0.f));
            if (ph == 1) {
#pragma unroll
              for (int e = 0; e < 4; ++e) gz[s][e] = x[s][e];
            }
          }
          // kept for the products over all rows: each column by the CTA that owns it (pairs of columns)
          float* keep = (ph == 1 ? p.Gz : p.dh) + row * d;
          if (has && (!SMALL || g < 4) && kb - 4 * c < d_lo + nd && ks1 * 16 > d_lo) {
#pragma unroll
            for (int s = 0; s < KC; ++s) {
              const int k = kb + 16 * s;
              if (ks0 + s < ks1 && k >= d_lo && k < d_lo + nd) *reinterpret_cast<float2*>(keep + k) = make_float2(x[s][0], x[s][1]);
              if (ks0 + s < ks1 && k + 2 >= d_lo && k + 2 < d_lo + nd) *reinterpret_cast<float2*>(keep + k + 2) = make_float2(x[s][2], x[s][3]);
            }
          }
        }
        const int n_here = ks1 - ks0 - s0;
        // the three terms of every value: rows g (hi | mid) and g + 8 (lo), or hi, mid and lo
        unsigned fa[KC][SMALL ? 4 : 6];
#pragma unroll
        for (int s = 0; s < KC; ++s) {
          unsigned h0, m0, l0, h1, m1, l1;
          if (s >= n_here) { x[s][0] = 0.f; x[s][1] = 0.f; x[s][2] = 0.f; x[s][3] = 0.f; }
          split3(x[s][0], x[s][1], h0, m0, l0);
          split3(x[s][2], x[s][3], h1, m1, l1);
          if constexpr (SMALL) { fa[s][0] = g < 4 ? h0 : m0; fa[s][1] = g < 4 ? l0 : 0u; fa[s][2] = g < 4 ? h1 : m1; fa[s][3] = g < 4 ? l1 : 0u; }
          else { fa[s][0] = h0; fa[s][1] = m0; fa[s][2] = h1; fa[s][3] = m1; fa[s][4] = l0; fa[s][5] = l1; }
        }
        // (several tiles only where one round covers the contraction)
#pragma unroll 1
        for (int t = 0; t < tiles; ++t) {
          if (t > 0) { acc0[0] = acc0[1] = acc0[2] = acc0[3] = 0.f; acc1[0] = acc1[1] = acc1[2] = acc1[3] = 0.f; }
          const int r = t * 8 + g < rows ? t * 8 + g : rows - 1;
          const unsigned char* wrow = wbase + ((size_t)r * stride + kb + 16 * s0) * 2;
#pragma unroll
          for (int s = 0; s < KC; ++s) {                       // (no branch around a product: steps beyond the stretch multiply zeros)
            const uint2 w = *reinterpret_cast<const uint2*>(wrow + (s < n_here ? s * 32 : 0));
            if constexpr (SMALL) bl_mma((s & 1) ? acc1 : acc0, fa[s][0], fa[s][1], fa[s][2], fa[s][3], w.x, w.y);
            else { bl_mma(acc0, fa[s][0], fa[s][1], fa[s][2], fa[s][3], w.x, w.y); bl_mma(acc1, fa[s][4], 0u, fa[s][5], 0u, w.x, w.y); }
          }
          red[(t * kBMma + warp) * 32 + lane] = make_float2((acc0[0] + acc0[2]) + (acc1[0] + acc1[2]), (acc0[1] + acc0[3]) + (acc1[1] + acc1[3]));
        }
#pragma unroll
        for (int s = 0; s < KC; ++s) xv[s] = xn[s];
      }
      if ((ph & 1) && norm && ks0 >= ks1) {                    // a warp without k-steps takes part in the barrier with zero sums
        if (c == 0) (reinterpret_cast<float2*>(smem + L.off_ssq) + (ph >> 1) * kBMma * 8)[warp * 8 + g] = make_float2(0.f, 0.f);
        b_sync();
      }
      b_sync();
      if (warp < tiles) {
        const int rl = warp * 8 + 2 * c;
        float y0 = 0.f, y1 = 0.f;
#pragma unroll
        for (int w = 0; w < kBMma; ++w) { const float2 v = red[(warp * kBMma + w) * 32 + lane]; y0 += v.x; y1 += v.y; }
        if (SMALL) { y0 += __shfl_xor_sync(0xffffffffu, y0, 16); y1 += __shfl_xor_sync(0xffffffffu, y1, 16); }
        if (has && rl < rows && (!SMALL || g < 4)) {
          if (ph == 0) bl_st2(p.dr + row * d + d_lo + rl, y0, y1);
          else if (ph == 1) {
            const float2 a = *reinterpret_cast<const float2*>(p.act + row * dff + f_lo + rl);
            bl_st2(p.dpre + row * dff + f_lo + rl, p.alpha * y0 * gelu_grad(a.x), p.alpha * y1 * gelu_grad(a.y));
          } else if (ph == 2) bl_st2(p.du + row * d + d_lo + rl, y0, y1);
          else bl_st2(p.dc + row * d + d_lo + rl, p.alpha * y0, p.alpha * y1);
        }
      }
    }
  }
}

}  // namespace

// Sequences per launch of this kernel for a batch of B, or 0 when it does not take the shape.
int bwd_leaf_slice(int B, int d, int H, int dff, int max_b) {
  if (B > max_b || d % 64 || d > 1024 || dff % 64) return 0;
  const int n_sub = ceil_div(B, 8), sub = ceil_div(B, n_sub);
  const BLoopLayout L = bloop_layout(d, dff, kB200Sms);
  if (sub * H > kB200Sms || L.nt_f > kBMma || L.nt_d > 1 || L.total > kB200SmemPerCta) return 0;
  return sub;
}

cudaError_t bwd_leaf_launch(const BwdLeafParams& p, cudaStream_t s) {
  BLoopLayout L = bloop_layout(p.d, p.dff, kB200Sms);
  const void* fn = p.B <= 4 ? reinterpret_cast<const void*>(&bwd_leaf_kernel<true>) : reinterpret_cast<const void*>(&bwd_leaf_kernel<false>);
  cudaError_t e = ensure_dynamic_smem(fn, (int)L.total);
  if (e != cudaSuccess) return e;
  BwdLeafParams pp = p;
  void* args[] = {(void*)&pp, (void*)&L};
  return cudaLaunchCooperativeKernel(fn, dim3(kB200Sms), dim3(kBThreads), args, L.total, s);
}

}  // namespace rt
