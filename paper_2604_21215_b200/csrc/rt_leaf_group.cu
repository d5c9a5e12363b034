// Leaf recurrence of several independent (layer, slice of sequences) jobs at once, bf16: the SMs are split into groups of
// equal size, one job each.  Used where jobs exist side by side: the layers of a stack (layer l works on a leaf that layer
// l-1 finished one launch earlier) and batches of more than 16 sequences (slices of at most 16).
//
// A token step is a chain of exchanges whose length does not depend on how many SMs take part, so a single job leaves
// 148 SMs waiting most of the time (rt_leaf_mma.cu).  Several jobs side by side fill the waits.  A group's weights (23 MB at
// d = 1024 over 37 SMs) do not stay on chip: every step streams them from L2 through a ring of bulk copies that keeps filling while the
// chain waits.  One SM takes 145 GB/s from L2 (all together 18 TB/s as long as the jobs' weights fit L2), but only in large pieces: a copy costs
// the copy unit about 90 ns whatever its size.  So the weights are packed once per call, in the order in which a CTA uses them.
//
// Exchanges and products are those of rt_leaf_mma.cu: words that carry their own step number for c, h, z and raw k|v, g behind a counter
// barrier of the group, m16n8k16 MMAs with the sequences as rows, K split over the eight MMA warps, one copy of the code for the four
// phases.  What differs: the weights come by pieces of 16 rows x d columns; a phase's activations are fetched once for all its pieces; seven
// attention warps own a (sequence, head) pair each, with a window of 16 queries in registers (two lanes per query), and fold the earlier
// positions of the leaf in when the window moves.
#include <cuda_bf16.h>
#include <string.h>

#include <type_traits>

#include "rt_kernels.h"
#include "rt_tc.cuh"

namespace rt {

namespace {

constexpr int kGMma = 8, kGAtt = 7;               // MMA warps, attention warps; the last warp issues the copies
constexpr int kGThreads = 512;
constexpr int kGMmaThreads = kGMma * 32;
constexpr int kGRegsMma = 184, kGRegsAtt = 72;    // (184 + 72) * 256 = 65536
constexpr int kWin = 16;
constexpr int kStStride = kHeadDim + 4;
constexpr int kMaxSlots = 16;
constexpr int kKP = 4;                            // blocks of 32 k per warp and stretch of d columns (d <= 1024)
constexpr int kPieceTiles = 2;                    // tiles of 8 weight rows per piece

// How a group of g CTAs shares the rows; a CTA's pieces of a step in order: W_o, W_up, W_down (stretch by stretch), W_k | W_v.
struct GroupShape { int max_nd, max_nf, nt_d, nt_f, nq, tiles; };      // upper bounds over the CTAs; tiles per step
__host__ __device__ inline GroupShape group_shape(int d, int dff, int g) {
  GroupShape s;
  s.max_nd = 2 * ((d / 2 + g - 1) / g);
  s.max_nf = 2 * ((dff / 2 + g - 1) / g);
  s.nt_d = (s.max_nd + 7) / 8; s.nt_f = (s.max_nf + 7) / 8; s.nq = (dff + d - 1) / d;
  s.tiles = s.nt_d + s.nt_f + s.nt_d * s.nq + 2 * s.nt_d;
  return s;
}

struct GroupLayout {
  int slots;                                      // ring entries
  GroupShape s;
  uint32_t off_red, off_ssq, off_hown, off_fin, off_state, off_ring, tile_bytes, total;
};

GroupLayout group_layout(int d, int dff, int mb, int g, size_t max_smem) {
  GroupLayout L;
  L.s = group_shape(d, dff, g);
  const int tiles = L.s.nt_f > 2 * L.s.nt_d ? L.s.nt_f : 2 * L.s.nt_d;
  uint32_t o = 512;
  auto take = [&](uint32_t n) { o = (o + 127) / 128 * 128; const uint32_t at = o; o += n; return at; };
  L.off_red = take((uint32_t)(kGMma * tiles * 32 * 8 * mb));
  L.off_ssq = take(kGMma * 16 * 4);
  L.off_hown = take((uint32_t)(16 * L.s.max_nd * 4));
  L.off_fin = take(kGAtt * 2048);
  L.off_state = take(kGAtt * kStStride * 4);
  L.off_ring = (o + 127) / 128 * 128;
  L.tile_bytes = (uint32_t)(8 * d * 2);           // [d / 32][8 rows][32]: the 16-byte fragment loads of eight lanes cover 128 bytes
  L.slots = max_smem > L.off_ring ? (int)((max_smem - L.off_ring) / (kPieceTiles * L.tile_bytes)) : 0;
  if (L.slots > kMaxSlots) L.slots = kMaxSlots;
  L.total = L.off_ring + (uint32_t)L.slots * kPieceTiles * L.tile_bytes;
  return L;
}

__device__ __forceinline__ float glo(unsigned u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float ghi(unsigned u) { return __uint_as_float(u & 0xffff0000u); }
__device__ __forceinline__ unsigned gpack(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const unsigned*>(&v);
}
__device__ __forceinline__ uint4 ld_two_words(const void* p) {
  unsigned long long a, b;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0,%1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
  return make_uint4((unsigned)a, (unsigned)(a >> 32), (unsigned)b, (unsigned)(b >> 32));
}
__device__ __forceinline__ uint4 ld_two_words_if(const void* p, unsigned on) {
  unsigned long long a = 0ull, b = 0ull;
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %3, 0;\n @q ld.relaxed.gpu.global.v2.u64 {%0,%1}, [%2];\n}"
               : "+l"(a), "+l"(b) : "l"(p), "r"(on) : "memory");
  return make_uint4((unsigned)a, (unsigned)(a >> 32), (unsigned)b, (unsigned)(b >> 32));
}
__device__ __forceinline__ uint4 ld_cg_if(const void* p, unsigned on) {
  uint4 w = make_uint4(0u, 0u, 0u, 0u);
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %5, 0;\n @q ld.global.cg.v4.u32 {%0,%1,%2,%3}, [%4];\n}"
               : "+r"(w.x), "+r"(w.y), "+r"(w.z), "+r"(w.w) : "l"(p), "r"(on) : "memory");
  return w;
}
__device__ __forceinline__ void st_flag(void* p, unsigned v, unsigned seq) {
  const unsigned long long w = ((unsigned long long)seq << 32) | v;
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ void st_flag2(void* p, unsigned a, unsigned b, unsigned seq) {
  const unsigned long long w0 = ((unsigned long long)seq << 32) | a, w1 = ((unsigned long long)seq << 32) | b;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1,%2};" ::"l"(p), "l"(w0), "l"(w1) : "memory");
}
__device__ __forceinline__ void gmma(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_sync_all() { asm volatile("bar.sync 1, %0;" ::"n"(kGMmaThreads) : "memory"); }

__device__ __noinline__ bool group_give_up(SyncArea* s, volatile int* s_abort, unsigned long long* t_start) {
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
// Waits for an mbarrier of this CTA (whole warp, one answer in all lanes).
__device__ __forceinline__ bool ring_wait(uint32_t bar, uint32_t parity, SyncArea* s, volatile int* s_abort) {
  unsigned spins = 0;
  unsigned long long t0 = 0;
  bool ok = true;
  while (ok && !mbar_try_wait(bar, parity))
    if ((++spins & 255u) == 0u && group_give_up(s, s_abort, &t0)) ok = false;
  return __all_sync(0xffffffffu, ok);
}
// Index of the 64-bit word {elements k, k + 1; step} of slot b (k even): [block of 32 k][16 slots][4 groups of 8 k][4 words].
__device__ __forceinline__ size_t w_idx(int b, int k) { return ((size_t)((k >> 5) * 16 + b) * 4 + ((k & 31) >> 3)) * 4 + ((k & 7) >> 1); }
// Byte offset of element k of slot b of g (packed bf16): [block of 32 k][16 slots][32 k].
__device__ __forceinline__ size_t g_off(int b, int k) { return ((size_t)((k >> 5) * 16 + b) << 6) + (size_t)(k & 31) * 2; }

struct GroupArgs {
  GroupCommon c;
  GroupJob job[kGroupJobs];
  int n_jobs, gsize;
};

// Packs one layer: CTA's tiles one after the other, a tile = 8 rows x d columns as [d / 32][8][32], rows beyond the CTA's own zero.
__global__ void __launch_bounds__(256) group_pack_kernel(GroupPackArgs a) {
  const GroupShape s = group_shape(a.d, a.dff, a.g);
  const int cta = blockIdx.x, tile = blockIdx.y, layer = blockIdx.z;
  const GroupPackLayer& w = a.layer[layer];
  const int d_lo = 2 * (int)((long long)(a.d / 2) * cta / a.g), nd = 2 * (int)((long long)(a.d / 2) * (cta + 1) / a.g) - d_lo;
  const int f_lo = 2 * (int)((long long)(a.dff / 2) * cta / a.g), nf = 2 * (int)((long long)(a.dff / 2) * (cta + 1) / a.g) - f_lo;
  int t = tile, rows = nd, row = d_lo, K = a.d, col = 0;
  const void* src;
  if (t < s.nt_d) src = w.w_o;
  else if ((t -= s.nt_d) < s.nt_f) { src = w.w_up; rows = nf; row = f_lo; }
  else if ((t -= s.nt_f) < s.nt_d * s.nq) { src = w.w_down; K = a.dff; col = (t / s.nt_d) * a.d; t %= s.nt_d; }
  else { t -= s.nt_d * s.nq; src = t < s.nt_d ? w.w_k : w.w_v; t %= s.nt_d; }
  const int n16 = a.d;                                         // 16-byte groups of a tile: 8 rows x d / 8
  uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(w.out) + ((size_t)cta * s.tiles + tile) * (size_t)(16 * a.d));
  for (int i = threadIdx.x; i < n16; i += 256) {
    const int r = i / (a.d / 8), k = (i % (a.d / 8)) * 8;       // consecutive threads read consecutive 16-byte groups of a row
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (t * 8 + r < rows && col + k < K)
      v = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(src) + (size_t)(row + t * 8 + r) * K + col + k);
    dst[(k >> 5) * 32 + r * 4 + ((k & 31) >> 3)] = v;
  }
}

// kQuad: tiles of weight rows a warp works on at a time (one or two pieces).
template <int MB, int kQuad>
__global__ void __launch_bounds__(kGThreads, 1) leaf_group_kernel(const __grid_constant__ GroupArgs a, const GroupLayout L) {
  extern __shared__ __align__(128) unsigned char smem[];
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem);
  const uint32_t full = smem_u32(smem + 64), empty = full + 8 * kMaxSlots;
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int G = a.gsize, job = blockIdx.x / G, cta = blockIdx.x - job * G;
  const GroupCommon& C = a.c;
  const GroupJob& J = a.job[job];
  SyncArea* const sync = C.sync;
  const int B = J.B, d = C.d, H = C.H, dff = C.dff, n = J.t1 - J.t0, pairs = B * H;
  // rows are dealt out in pairs so that a published word (two consecutive rows) has one owner
  const int d_lo = 2 * (int)((long long)(d / 2) * cta / G), nd = 2 * (int)((long long)(d / 2) * (cta + 1) / G) - d_lo;
  const int f_lo = 2 * (int)((long long)(dff / 2) * cta / G), nf = 2 * (int)((long long)(dff / 2) * (cta + 1) / G) - f_lo;
  const int nt_d = L.s.nt_d, nt_f = L.s.nt_f, nq = L.s.nq;     // (bounds: a CTA with fewer rows multiplies zero rows)
  unsigned char* const wd = J.words;
  unsigned* const counter = reinterpret_cast<unsigned*>(wd);
  const size_t vec_bytes = (size_t)16 * (d / 2) * 8;
  unsigned char *const w_c = wd + 256, *const w_h = w_c + vec_bytes, *const w_z = w_h + vec_bytes, *const w_g = w_z + vec_bytes, *const w_kv = w_g + (size_t)16 * dff * 2;

  if (tid == 0) {
    *s_abort = *reinterpret_cast<volatile unsigned*>(&sync->abort_flag) ? 1 : 0;
#pragma unroll 1
    for (int i = 0; i < L.slots; ++i) { mbar_init(full + 8 * i, 1); mbar_init(empty + 8 * i, kGMma); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  if (warp >= kGMma) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kGRegsAtt));
    if (warp == kGMma + kGAtt) {
      // ------------------------------ weights, in the order the products use them, across steps ------------------------------
      int slot = 0;
      uint32_t par = 0;
      bool ok = true, fresh = true;                            // fresh: first round of the ring, nothing to wait for
      const unsigned char* src = reinterpret_cast<const unsigned char*>(J.packed) + (size_t)cta * L.s.tiles * L.tile_bytes;
      // (one copy of the code, rolled: what this warp runs shares the instruction cache with the chain)
#pragma unroll 1
      for (int j = 0; j < n && ok; ++j) {
        const unsigned char* at = src;
#pragma unroll 1
        for (int r = 0; r < nq + 3 && ok; ++r) {               // W_o, W_up, the stretches of W_down, W_k | W_v
          int left = r == 1 ? nt_f : r == nq + 2 ? 2 * nt_d : nt_d;
#pragma unroll 1
          while (left > 0) {
            if (!fresh) ok = ring_wait(empty + 8 * slot, par, sync, s_abort);
            if (!ok) break;
            const uint32_t bar = full + 8 * slot, dst = smem_u32(smem + L.off_ring) + (uint32_t)slot * kPieceTiles * L.tile_bytes;
            const uint32_t bytes = (uint32_t)(left < kPieceTiles ? left : kPieceTiles) * L.tile_bytes;
            expect_tx_elect(bar, bytes);
            asm volatile("{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n @e cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n}"
                         ::"r"(dst), "l"(at), "r"(bytes), "r"(bar) : "memory");
            at += bytes;
            left -= kPieceTiles;
            if (++slot == L.slots) { slot = 0; if (!fresh) par ^= 1; fresh = false; }
          }
        }
      }
      if (!ok)                                                 // gave up: let the copies in flight land (bounded)
#pragma unroll 1
        for (int i = 0; i < L.slots; ++i)
#pragma unroll 1
          for (int spins = 0; spins < (1 << 13); ++spins) mbar_try_wait(full + 8 * i, 0);
      return;
    }
    // ------------------------------ attention: one (sequence, head) pair per warp ------------------------------
    // Lanes as dimensions (two each) for what the chain waits for: the pair of position j finishes query j + 1, whose value goes out.
    // Lanes as queries (two per query, 32 dimensions each) for the rest of the window, which absorbs the pair while the mat-vecs of the next
    // step run.  When a window opens, its queries first absorb the earlier positions, from key0 on, from the cache.
    const int aw = warp - kGMma, pair = cta + aw * G;
    if (pair < pairs) {
      const int b = pair / H, h = pair % H, bc = J.b0 + b;
      const __nv_bfloat16 *q = reinterpret_cast<const __nv_bfloat16*>(J.q), *g_k = reinterpret_cast<const __nv_bfloat16*>(J.g_k);
      __nv_bfloat16 *kc = reinterpret_cast<__nv_bfloat16*>(J.k_cache), *vc = reinterpret_cast<__nv_bfloat16*>(J.v_cache);
      const size_t qcol = (size_t)bc * d + h * kHeadDim, qrow = (size_t)C.Bs * d;      // a position's row of q, state and caches
      const float slope = J.alibi ? J.alibi[h] * kLog2e : 0.f;
      float* fin = reinterpret_cast<float*>(smem + L.off_fin + aw * 2048);            // four pairs (k[64], v[64])
      float* st = reinterpret_cast<float*>(smem + L.off_state) + aw * kStStride;      // o, m, l of the query that is finished next
      unsigned char* const c_at = w_c + w_idx(b, h * kHeadDim + 2 * lane) * 8;
      const unsigned char* const kv_at = w_kv + ((size_t)b * 2 * d + h * kHeadDim + 2 * lane) * 8;
      const bool qkn = (C.norm_flags & RT_NORM_QK) != 0;
      const float gk0 = qkn ? gain_at(g_k, h * kHeadDim + 2 * lane) : 1.f, gk1 = qkn ? gain_at(g_k, h * kHeadDim + 2 * lane + 1) : 1.f;
      const int qi = lane >> 1, e0 = (lane & 1) * 32;          // query of the window, dimensions of this lane
      unsigned qr[16];                                         // its query as packed bf16
      float o[32], m = 0.f, l = 1.f;
      int w0 = 0;                                              // first position (in the leaf) of the window
      auto fold = [&](const float* kf, int dist) {             // absorb the pair at kf (k[64], v[64] fp32)
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
          const float4 kk = *reinterpret_cast<const float4*>(kf + e0 + e);
          s0 = fmaf(glo(qr[e / 2]), kk.x, s0); s1 = fmaf(ghi(qr[e / 2]), kk.y, s1);
          s0 = fmaf(glo(qr[e / 2 + 1]), kk.z, s0); s1 = fmaf(ghi(qr[e / 2 + 1]), kk.w, s1);
        }
        float s = s0 + s1;
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s = s * C.scale_log2 - slope * (float)dist;
        const float mn = fmaxf(m, s), corr = exp2f(m - mn), pj = exp2f(s - mn);
        m = mn; l = l * corr + pj;
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
          const float4 vv = *reinterpret_cast<const float4*>(kf + kHeadDim + e0 + e);
          o[e] = fmaf(o[e], corr, pj * vv.x); o[e + 1] = fmaf(o[e + 1], corr, pj * vv.y);
          o[e + 2] = fmaf(o[e + 2], corr, pj * vv.z); o[e + 3] = fmaf(o[e + 3], corr, pj * vv.w);
        }
      };
      auto leave_state = [&]() {
#pragma unroll
        for (int e = 0; e < 32; e += 4) *reinterpret_cast<float4*>(st + e0 + e) = make_float4(o[e], o[e + 1], o[e + 2], o[e + 3]);
        if (e0 == 0) { st[kHeadDim] = m; st[kHeadDim + 1] = l; }
      };
      // One copy of everything long (what these warps run shares the instruction cache with the chain): iteration j = -1 opens the
      // first window, iteration j >= 0 finishes query j + 1 and absorbs pair j -- or opens the next window and absorbs every earlier pair.
#pragma unroll 1
      for (int j = -1; j < n; ++j) {
        const unsigned seq = J.steps + (unsigned)(j + 1);      // step that reveals position t0 + j
        unsigned kw[4], vw[4];
        kw[0] = vw[0] = 0u;
        if (j >= 0) {
          float q0 = 0.f, q1 = 0.f;
          if (j + 1 < n) {
            const unsigned qw = *reinterpret_cast<const unsigned*>(q + (size_t)(J.t0 - J.row_off + j + 1) * qrow + qcol + 2 * lane);
            q0 = glo(qw); q1 = ghi(qw);
          }
          uint4 ka, va;
          {
            unsigned spins = 0;
            unsigned long long t0 = 0;
            while (true) {
              ka = ld_two_words(kv_at);
              va = ld_two_words(kv_at + (size_t)d * 8);
              if (__all_sync(0xffffffffu, ka.y == seq && ka.w == seq && va.y == seq && va.w == seq)) break;
              if ((++spins & 63u) == 0u && __any_sync(0xffffffffu, group_give_up(sync, s_abort, &t0))) break;
            }
          }
          const float2 kr = make_float2(__uint_as_float(ka.x), __uint_as_float(ka.z)), vr = make_float2(__uint_as_float(va.x), __uint_as_float(va.z));
          // Eq. (1): qkRMS over the head, then the storage rounding the cache applies
          const float rk = qkn ? rsqrtf(warp_sum(kr.x * kr.x + kr.y * kr.y) * (1.0f / kHeadDim) + C.eps) : 1.0f;
          const unsigned kq = gpack(kr.x * rk * gk0, kr.y * rk * gk1), vq = gpack(vr.x, vr.y);
          const float k0 = glo(kq), k1 = ghi(kq), v0 = glo(vq), v1 = ghi(vq);
          if (j + 1 < n) {
            const float s = warp_sum(q0 * k0 + q1 * k1) * C.scale_log2 - slope;
            const float mo = st[kHeadDim], mn = fmaxf(mo, s), corr = exp2f(mo - mn), pj = exp2f(s - mn);
            const float il = 1.0f / (st[kHeadDim + 1] * corr + pj);
            const float2 oo = *reinterpret_cast<const float2*>(st + 2 * lane);
            st_flag(c_at, gpack((oo.x * corr + pj * v0) * il, (oo.y * corr + pj * v1) * il), seq + 1u);
          }
          const size_t crow = (size_t)(J.t0 + j) * qrow + qcol + 2 * lane;
          *reinterpret_cast<unsigned*>(kc + crow) = kq;
          *reinterpret_cast<unsigned*>(vc + crow) = vq;
          if (j + 2 >= n) continue;
          kw[0] = kq; vw[0] = vq;
          __syncwarp();
        }
        const bool open = j < 0 || j + 2 == w0 + kWin;
        const int key1 = J.t0 + j + 1;
        int key = J.t0 + j;                                    // pairs [key, key1) to absorb
        auto fetch = [&](int j0) {                             // four pairs in flight
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const size_t kr = (size_t)min(j0 + u, key1 - 1) * qrow + qcol + 2 * lane;
            kw[u] = __ldcg(reinterpret_cast<const unsigned*>(kc + kr)); vw[u] = __ldcg(reinterpret_cast<const unsigned*>(vc + kr));
          }
        };
        if (open) {
          w0 = j < 0 ? 0 : j + 2;
          const int i = min(w0 + qi, n - 1);
          const size_t row = (size_t)(J.t0 - J.row_off + i), at = row * qrow + qcol + e0;
#pragma unroll
          for (int e = 0; e < 32; e += 8) {
            const uint4 w = *reinterpret_cast<const uint4*>(q + at + e);
            qr[e / 2] = w.x; qr[e / 2 + 1] = w.y; qr[e / 2 + 2] = w.z; qr[e / 2 + 3] = w.w;
          }
#pragma unroll
          for (int e = 0; e < 32; e += 4) {
            const float4 w = *reinterpret_cast<const float4*>(J.st_o + at + e);
            o[e] = w.x; o[e + 1] = w.y; o[e + 2] = w.z; o[e + 3] = w.w;
          }
          m = J.st_m[(row * C.Bs + bc) * H + h]; l = J.st_l[(row * C.Bs + bc) * H + h];
          key = J.key0;
          if (key < key1) fetch(key);
        }
#pragma unroll 1
        for (; key < key1; key += 4) {
          __syncwarp();
          const int here = min(4, key1 - key);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (u < here) {
              *reinterpret_cast<float2*>(fin + u * 128 + 2 * lane) = make_float2(glo(kw[u]), ghi(kw[u]));
              *reinterpret_cast<float2*>(fin + u * 128 + kHeadDim + 2 * lane) = make_float2(glo(vw[u]), ghi(vw[u]));
            }
          }
          __syncwarp();
          if (key + 4 < key1) fetch(key + 4);
#pragma unroll 1
          for (int u = 0; u < here; ++u) fold(fin + u * 128, J.t0 + w0 + qi - key - u);
        }
        if (j < 0) {
          if (qi == 0) leave_state();
          __syncwarp();
          const float il = 1.f / st[kHeadDim + 1];
          const float2 oo = *reinterpret_cast<const float2*>(st + 2 * lane);
          st_flag(c_at, gpack(oo.x * il, oo.y * il), J.steps + 1u);
          __syncwarp();
        }
        if (w0 + qi == j + 2) leave_state();
        __syncwarp();
      }
    }
    return;
  }

  // ------------------------------ MMA warps (after a wait that ran out they go on to the end: barriers need every warp) ------------------------------
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kGRegsMma));
  using Part = typename std::conditional<MB == 2, float4, float2>::type;
  Part* red = reinterpret_cast<Part*>(smem + L.off_red);       // [tile][warp][lane]
  float* ssq_red = reinterpret_cast<float*>(smem + L.off_ssq);
  float* hown = reinterpret_cast<float*>(smem + L.off_hown);
  const int g = lane >> 2, c = lane & 3;
  const bool pre = (C.norm_flags & RT_NORM_PRE) != 0, kv_norm = pre && !(C.norm_flags & RT_NORM_SKIP_Z);
  const float inv_d = 1.0f / (float)d;
  const bool has0 = g < B, has1 = MB == 2 && g + 8 < B;
  const int nkp = d >> 5, per = (nkp + kGMma - 1) / kGMma;
  const int n_kp = max(0, min(per, nkp - warp * per));         // this warp's blocks of 32 k in a stretch of d
  const int kp0 = n_kp > 0 ? warp * per : 0;                   // (a warp without any multiplies the first one by zeros)
  const __nv_bfloat16* x = reinterpret_cast<const __nv_bfloat16*>(J.x);
  __nv_bfloat16* z = reinterpret_cast<__nv_bfloat16*>(J.z);
  unsigned target = J.steps * (unsigned)G;
  int slot = 0;
  uint32_t par = 0;
  const unsigned char* const ring = smem + L.off_ring + g * 64 + c * 16 + kp0 * 512;

#pragma unroll 1
  for (int j = 0; j < n; ++j) {
    const unsigned seq = J.steps + (unsigned)j + 1u;
    const size_t t = (size_t)(J.t0 + j);
#pragma unroll 1
    for (int ph = 0; ph < 4; ++ph) {                           // 0: W_o   1: W_up   2: W_down   3: W_k | W_v
      const int rows = ph == 1 ? nf : nd, tiles = ph == 1 ? nt_f : ph == 3 ? 2 * nt_d : nt_d;
      const bool want_ssq = ph == 1 ? pre : ph == 3 && kv_norm;
      uint4 av[kKP][MB], an[kKP][MB];
      float sq0 = 0.f, sq1 = 0.f;
      unsigned xw0 = 0, xw1 = 0;
      if (ph == 0 && warp < tiles && warp * 8 + 2 * c < nd) {  // x_t for the residual, fetched before the wait
        if (has0) xw0 = *reinterpret_cast<const unsigned*>(x + (size_t)g * J.x_bs + t * J.x_ts + d_lo + warp * 8 + 2 * c);
        if (has1) xw1 = *reinterpret_cast<const unsigned*>(x + (size_t)(g + 8) * J.x_bs + t * J.x_ts + d_lo + warp * 8 + 2 * c);
      }
      auto load_g = [&](uint4 (&v)[kKP][MB], int q) {          // stretch q of g
        const unsigned char* base = w_g + (size_t)(q * nkp + kp0) * 1024 + g * 64 + c * 16;
        const int lim = min(n_kp, (dff >> 5) - q * nkp - kp0);
#pragma unroll
        for (int i = 0; i < kKP; ++i)
#pragma unroll
          for (int r = 0; r < MB; ++r) v[i][r] = ld_cg_if(base + (size_t)(i < lim ? i : 0) * 1024 + r * 512, i < lim && (r ? has1 : has0) ? 1u : 0u);
      };
      if (ph == 2) {
        // every CTA's slice of g must be there before anyone multiplies by W_down
        target += (unsigned)G;
        if (tid == 0) {
          unsigned spins = 0;
          unsigned long long t0 = 0;
          while (ld_acquire_u32(counter) < target)
            if ((++spins & 255u) == 0u && group_give_up(sync, s_abort, &t0)) break;
        }
        mma_sync_all();
        load_g(av, 0);
      } else {
        const unsigned char* base = (ph == 0 ? w_c : ph == 1 ? w_h : w_z) + ((size_t)kp0 * 16 + g) * 128 + c * 32;
        unsigned need[MB];
#pragma unroll
        for (int r = 0; r < MB; ++r) need[r] = (r ? has1 : has0) ? (1u << n_kp) - 1u : 0u;
#pragma unroll
        for (int i = 0; i < kKP; ++i)
#pragma unroll
          for (int r = 0; r < MB; ++r) av[i][r] = make_uint4(0u, 0u, 0u, 0u);
        unsigned spins = 0;
        unsigned long long t0 = 0;
        // more than eight sequences: one pair of words first; rounds over all of them would crowd out the attention warps' own loads (33 -> 28 us a step)
        while (MB == 2 && n_kp > 0) {
          const uint4 w = ld_two_words_if(base, has0 ? 1u : 0u);
          if (__all_sync(0xffffffffu, !has0 || (w.y == seq && w.w == seq))) break;
          if ((++spins & 63u) == 0u && __any_sync(0xffffffffu, group_give_up(sync, s_abort, &t0))) break;
        }
        while (true) {
          uint4 wa[kKP][MB], wb[kKP][MB];                      // all outstanding words are on their way before any is looked at
#pragma unroll
          for (int i = 0; i < kKP; ++i)
#pragma unroll
            for (int r = 0; r < MB; ++r) {
              const unsigned char* at = base + (size_t)(i < n_kp ? i : 0) * 2048 + r * 1024;
              wa[i][r] = ld_two_words_if(at, (need[r] >> i) & 1u);
              wb[i][r] = ld_two_words_if(at + 16, (need[r] >> i) & 1u);
            }
          unsigned left = 0;
#pragma unroll
          for (int r = 0; r < MB; ++r) {
#pragma unroll
            for (int i = 0; i < kKP; ++i) {
              const bool ok = ((need[r] >> i) & 1u) && wa[i][r].y == seq && wa[i][r].w == seq && wb[i][r].y == seq && wb[i][r].w == seq;
              if (ok) { av[i][r] = make_uint4(wa[i][r].x, wa[i][r].z, wb[i][r].x, wb[i][r].z); need[r] &= ~(1u << i); }
            }
            left |= need[r];
          }
          if (__all_sync(0xffffffffu, left == 0u)) break;
          if ((++spins & 63u) == 0u && __any_sync(0xffffffffu, group_give_up(sync, s_abort, &t0))) break;
        }
        if (want_ssq) {
          const __nv_bfloat16* gain = reinterpret_cast<const __nv_bfloat16*>(ph == 1 ? J.g_mlp : J.g_kv);
#pragma unroll
          for (int i = 0; i < kKP; ++i) {
#pragma unroll
            for (int r = 0; r < MB; ++r) {
              uint4& v = av[i][r];
              const float e0 = glo(v.x), e1 = ghi(v.x), e2 = glo(v.y), e3 = ghi(v.y), e4 = glo(v.z), e5 = ghi(v.z), e6 = glo(v.w), e7 = ghi(v.w);
              const float s = ((e0 * e0 + e1 * e1) + (e2 * e2 + e3 * e3)) + ((e4 * e4 + e5 * e5) + (e6 * e6 + e7 * e7));
              if (r) sq1 += s; else sq0 += s;
              if (gain) {
                const uint4 gv = *reinterpret_cast<const uint4*>(gain + (kp0 + (i < n_kp ? i : 0)) * 32 + 8 * c);
                v.x = gpack(e0 * glo(gv.x), e1 * ghi(gv.x)); v.y = gpack(e2 * glo(gv.y), e3 * ghi(gv.y));
                v.z = gpack(e4 * glo(gv.z), e5 * ghi(gv.z)); v.w = gpack(e6 * glo(gv.w), e7 * ghi(gv.w));
              }
            }
          }
          sq0 += __shfl_xor_sync(0xffffffffu, sq0, 1); sq0 += __shfl_xor_sync(0xffffffffu, sq0, 2);
          sq1 += __shfl_xor_sync(0xffffffffu, sq1, 1); sq1 += __shfl_xor_sync(0xffffffffu, sq1, 2);
          if (c == 0) { ssq_red[warp * 16 + g] = sq0; ssq_red[warp * 16 + 8 + g] = sq1; }
        }
      }
      // ---- products: one or two pieces of the ring at a time ----
      const int n_q = ph == 2 ? nq : 1;
      const bool keep = tiles <= kQuad;                        // the sums of all stretches stay in registers
      float acc[kQuad][2][4];
#pragma unroll 1
      for (int q = 0; q < n_q; ++q) {
        if (q + 1 < n_q) load_g(an, q + 1);
#pragma unroll 1
        for (int ti = 0; ti < tiles; ti += kQuad) {
          const int slot2 = slot + 1 == L.slots ? 0 : slot + 1;
          const bool two = kQuad > kPieceTiles && ti + kPieceTiles < tiles;
          ring_wait(full + 8 * slot, par, sync, s_abort);
          if (two) ring_wait(full + 8 * slot2, slot2 ? par : par ^ 1, sync, s_abort);
          const unsigned char* w0 = ring + (size_t)slot * kPieceTiles * L.tile_bytes;
          const unsigned char* w1 = ring + (size_t)(two ? slot2 : slot) * kPieceTiles * L.tile_bytes;      // (products of tiles that do not exist are not used)
          if (q == 0 || !keep) {
#pragma unroll
            for (int u = 0; u < kQuad; ++u)
#pragma unroll
              for (int e = 0; e < 4; ++e) { acc[u][0][e] = 0.f; acc[u][1][e] = 0.f; }
          }
#pragma unroll
          for (int i = 0; i < kKP; ++i) {                      // (no branch around a product: blocks beyond the stretch multiply zeros)
            const int at = i < n_kp ? i * 512 : 0;
            uint4 bw[kQuad];
#pragma unroll
            for (int u = 0; u < kQuad; ++u) bw[u] = *reinterpret_cast<const uint4*>((u < kPieceTiles ? w0 : w1) + (size_t)(u & 1) * L.tile_bytes + at);
#pragma unroll
            for (int u = 0; u < kQuad; ++u)
              gmma(acc[u][0], av[i][0].x, MB == 2 ? av[i][MB - 1].x : 0u, av[i][0].y, MB == 2 ? av[i][MB - 1].y : 0u, bw[u].x, bw[u].y);
#pragma unroll
            for (int u = 0; u < kQuad; ++u)
              gmma(acc[u][1], av[i][0].z, MB == 2 ? av[i][MB - 1].z : 0u, av[i][0].w, MB == 2 ? av[i][MB - 1].w : 0u, bw[u].z, bw[u].w);
          }
          __syncwarp();
          if (lane == 0) { mbar_arrive(empty + 8 * slot); if (two) mbar_arrive(empty + 8 * slot2); }
          for (int k = 0; k < (two ? 2 : 1); ++k)
            if (++slot == L.slots) { slot = 0; par ^= 1; }
          if (keep && q + 1 < n_q) continue;
#pragma unroll
          for (int u = 0; u < kQuad; ++u) {
            if (ti + u < tiles) {
              Part* dst = red + ((ti + u) * kGMma + warp) * 32 + lane;
              Part v;
              v.x = acc[u][0][0] + acc[u][1][0]; v.y = acc[u][0][1] + acc[u][1][1];
              if constexpr (MB == 2) { v.z = acc[u][0][2] + acc[u][1][2]; v.w = acc[u][0][3] + acc[u][1][3]; }
              if (q > 0 && !keep) {
                const Part old = *dst;
                v.x += old.x; v.y += old.y;
                if constexpr (MB == 2) { v.z += old.z; v.w += old.w; }
              }
              *dst = v;
            }
          }
        }
#pragma unroll
        for (int i = 0; i < kKP; ++i)
#pragma unroll
          for (int r = 0; r < MB; ++r) av[i][r] = an[i][r];
      }
      mma_sync_all();
      // ---- sums over the eight warps; warp w finishes the tiles w, w + 8, ... ----
      float rs0 = 1.0f, rs1 = 1.0f;
      if (want_ssq) {
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int w = 0; w < kGMma; ++w) { s0 += ssq_red[w * 16 + g]; if (MB == 2) s1 += ssq_red[w * 16 + 8 + g]; }
        rs0 = rsqrtf(s0 * inv_d + C.eps);
        if (MB == 2) rs1 = rsqrtf(s1 * inv_d + C.eps);
      }
#pragma unroll 1
      for (int ti = warp; ti < tiles; ti += kGMma) {
        const bool second = ph == 3 && ti >= nt_d;
        const int rl = (second ? ti - nt_d : ti) * 8 + 2 * c;
        float y0 = 0.f, y1 = 0.f, y2 = 0.f, y3 = 0.f;
#pragma unroll
        for (int w = 0; w < kGMma; ++w) {
          const Part v = red[(ti * kGMma + w) * 32 + lane];
          y0 += v.x; y1 += v.y;
          if constexpr (MB == 2) { y2 += v.z; y3 += v.w; }
        }
        if (rl >= rows) continue;
        if (ph == 0) {                                         // h = x_t + alpha W_o c_t
          if (has0) {
            const float h0 = glo(xw0) + C.alpha * y0, h1 = ghi(xw0) + C.alpha * y1;
            *reinterpret_cast<float2*>(hown + g * L.s.max_nd + rl) = make_float2(h0, h1);
            st_flag(w_h + w_idx(g, d_lo + rl) * 8, gpack(h0, h1), seq);
          }
          if (has1) {
            const float h0 = glo(xw1) + C.alpha * y2, h1 = ghi(xw1) + C.alpha * y3;
            *reinterpret_cast<float2*>(hown + (g + 8) * L.s.max_nd + rl) = make_float2(h0, h1);
            st_flag(w_h + w_idx(g + 8, d_lo + rl) * 8, gpack(h0, h1), seq);
          }
        } else if (ph == 1) {                                  // g = GELU(W_up RMS(h)), packed bf16
          auto gelu = [](float v) { return 0.5f * v * (1.0f + erff(v * 0.70710678118654752f)); };
          if (has0) *reinterpret_cast<unsigned*>(w_g + g_off(g, f_lo + rl)) = gpack(gelu(y0 * rs0), gelu(y1 * rs0));
          if (has1) *reinterpret_cast<unsigned*>(w_g + g_off(g + 8, f_lo + rl)) = gpack(gelu(y2 * rs1), gelu(y3 * rs1));
        } else if (ph == 2) {                                  // z_t = h + alpha W_down g   (layer output)
#pragma unroll
          for (int r = 0; r < MB; ++r) {
            const int b = g + 8 * r;
            if (!(r ? has1 : has0)) continue;
            const float2 h = *reinterpret_cast<const float2*>(hown + b * L.s.max_nd + rl);
            const unsigned zw = gpack(h.x + C.alpha * (r ? y2 : y0), h.y + C.alpha * (r ? y3 : y1));
            st_flag(w_z + w_idx(b, d_lo + rl) * 8, zw, seq);
            *reinterpret_cast<unsigned*>(z + (size_t)b * J.z_bs + t * J.z_ts + d_lo + rl) = zw;
          }
        } else {                                               // raw k_t, v_t from RMS(z_t): Eqs. (1)-(2) before qkRMS
          const size_t col = (size_t)(second ? d : 0) + d_lo + rl;
          if (has0) st_flag2(w_kv + ((size_t)g * 2 * d + col) * 8, __float_as_uint(y0 * rs0), __float_as_uint(y1 * rs0), seq);
          if (has1) st_flag2(w_kv + ((size_t)(g + 8) * 2 * d + col) * 8, __float_as_uint(y2 * rs1), __float_as_uint(y3 * rs1), seq);
        }
      }
      mma_sync_all();                                          // red may be written again
      if (ph == 1 && tid == 0) red_release_add_u32(counter, 1u);   // (cumulative over what the barrier ordered before it)
    }
  }
}

}  // namespace

size_t leaf_group_words_bytes(int d, int dff) { return align_up(256 + (size_t)3 * 16 * (d / 2) * 8 + (size_t)16 * dff * 2 + (size_t)16 * 2 * d * 8, 256); }
size_t leaf_group_packed_bytes(int d, int dff, int places) {
  const int g = kB200Sms / places;
  return align_up((size_t)g * group_shape(d, dff, g).tiles * 16 * d, 256);
}

// Whether jobs of B sequences run on groups of 148 / places SMs (pure arithmetic).
bool leaf_group_shape(int B, int d, int H, int dff, int places, size_t max_smem) {
  if (B < 1 || B > 16 || places < 1 || places > kGroupJobs || d % 64 || d > 1024 || dff % 32 || dff > 8 * d) return false;
  const int g = kB200Sms / places;
  if (B * H > kGAtt * g || group_shape(d, dff, g).nt_d > kGMma) return false;
  return group_layout(d, dff, B > 8 ? 2 : 1, g, max_smem).slots >= 4;
}

cudaError_t leaf_group_pack(const GroupPackLayer* layers, int n, int d, int dff, int places, cudaStream_t s) {
  const int g = kB200Sms / places;
  for (int l0 = 0; l0 < n; l0 += kGroupPackLayers) {
    GroupPackArgs a;
    memset(&a, 0, sizeof(a));
    a.d = d; a.dff = dff; a.g = g;
    const int here = n - l0 < kGroupPackLayers ? n - l0 : kGroupPackLayers;
    for (int i = 0; i < here; ++i) a.layer[i] = layers[l0 + i];
    group_pack_kernel<<<dim3(g, group_shape(d, dff, g).tiles, here), 256, 0, s>>>(a);
  }
  return cudaGetLastError();
}

cudaError_t leaf_group_launch(const GroupCommon& c, const GroupJob* jobs, int n_jobs, int places, cudaStream_t s) {
  GroupArgs a;
  memset(&a, 0, sizeof(a));
  a.c = c; a.n_jobs = n_jobs; a.gsize = kB200Sms / places;
  int most = 0;
  for (int i = 0; i < n_jobs; ++i) { a.job[i] = jobs[i]; most = jobs[i].B > most ? jobs[i].B : most; }
  const int mb = most > 8 ? 2 : 1;
  GroupLayout L = group_layout(c.d, c.dff, mb, a.gsize, kB200SmemPerCta);
  // Two pieces at a time overlap more loads and products, but the longer code costs every phase (the step runs each instruction once or a few
  // times): at 37 SMs per group, d = 1024, B = 16 a step takes 29.5 us so against 31.3; at d = 768, B = 14 21.4 against 20.3, at d = 256 17.5 against 15.9.
  const bool wide = mb == 2 && L.s.nt_f > 12;
  const void* fn = wide ? (const void*)&leaf_group_kernel<2, 2 * kPieceTiles>
                        : mb == 2 ? (const void*)&leaf_group_kernel<2, kPieceTiles> : (const void*)&leaf_group_kernel<1, kPieceTiles>;
  cudaError_t e = ensure_dynamic_smem(fn, (int)L.total);
  if (e != cudaSuccess) return e;
  void* args[] = {(void*)&a, (void*)&L};
  return cudaLaunchCooperativeKernel(fn, dim3(a.gsize * n_jobs), dim3(kGThreads), args, L.total, s);
}

}  // namespace rt
