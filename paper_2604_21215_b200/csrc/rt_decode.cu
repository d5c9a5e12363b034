// One decode step (bf16 storage, up to 16 sequences per launch) through up to kDecMaxLayers layers as ONE cooperative kernel.
//
// A decode step reads every weight and the whole cache once and does little arithmetic with them, so its floor is the HBM
// time of those bytes; what kept the launch-per-phase form away from it was the chain of phases (launches, then reading
// weights that nobody had asked for yet).  Here one CTA per SM stays for all layers:
//   * each CTA owns a slice of the rows of every matrix.  A layer's slices fill shared memory; as soon as a slice has been
//     used, the bulk copies of the NEXT layer's slice go into its place, so weights stream from HBM under the other
//     phases.  (Wq and Wo share a place, and the Wk, Wv places alternate between layers, because a layer's persistent
//     pair is computed one phase later, next to the following layer's projections of the same vector.)
//   * while the mat-vec phases run, helper warps ask L2 for the cache rows that their chunk of the next layer's
//     attention will read.
//   * phases hand their vectors over through L2 words that are their own flags: the exchange area is filled with
//     0xFFFFFFFF (a NaN pattern no conversion produces) before the launch, every word is written once, and a consumer
//     polls the words themselves.  No barrier across CTAs, no second round trip.
// The vectors c, h, g, z travel as bf16, up to 16 sequences a launch, or (FULL) as fp32, up to eight: a value is then multiplied as three
// bf16 terms whose sum it is (24 bits), the first two in the rows that the other eight sequences would take, the third in a second MMA.
// Phases of layer l (K split over warps, partial sums through shared memory; sequences are the MMA's rows):
//   1. x = z^{l-1}: q, k~, v~ of layer l and the raw persistent k, v of layer l-1 (raw fp32 words)
//   2. attention over the cache: warp = (four heads, chunk of positions), Algorithm 2 per group of eight positions;
//      the warps of a CTA merge through shared memory, one partial state per (four heads, CTA) goes out
//   3. the CTA that owns a (sequence, head) pair folds the partial states into the seed of the temporary pair -> c
//   4. h = x + alpha W_o c    5. g = GELU(W_up RMS(h))    6. z = h + alpha W_down g
// and after the last layer one more phase 1 for its persistent pair.
#include <cuda_bf16.h>
#include <string.h>

#include "rt_kernels.h"
#include "rt_tc.cuh"

namespace rt {

namespace {

constexpr int kDecThreads = 512, kDecWarps = kDecThreads / 32;
constexpr int kMvWarps = 8;                      // warps that split K in the d-wide products; W_down splits over all 16
constexpr int kKeys = 8;                         // positions per round of the attention
constexpr int kPartStride = 68;                  // floats of one partial state: o[64], m, l, padding
constexpr unsigned kEmpty = 0xffffffffu;         // word that has not been written yet

struct DecLayout {
  int max_nd, max_nf, stride_d, stride_f;        // rows per CTA (upper bounds), row strides in elements
  int has_d, has_up, has_dn;                     // which slices live in shared memory (otherwise they are read from L2)
  unsigned off_red, off_ssq, off_hown, off_zown, off_mrg, off_q, off_kv, off_up, off_dn, total;
};

// Row strides leave 64 bytes modulo 128: the two rows that a quarter warp reads with 16-byte loads fall into different halves of the banks.
inline int row_stride(int K) { return (K * 2) % 128 == 64 ? K : K + 32; }

DecLayout dec_layout(int d, int dff, int grid, size_t max_smem) {
  DecLayout L;
  L.max_nd = 2 * ceil_div(d / 2, grid);
  L.max_nf = 2 * ceil_div(dff / 2, grid);
  L.stride_d = row_stride(d);
  L.stride_f = row_stride(dff);
  const int nt_d = ceil_div(L.max_nd, 8), nt_f = ceil_div(L.max_nf, 8);
  size_t o = 128;                                              // abort flag, mbarriers
  size_t red = (size_t)kMvWarps * (5 * nt_d > nt_f ? 5 * nt_d : nt_f) * 512;
  const size_t red_dn = (size_t)kDecWarps * nt_d * 512, part = (size_t)kDecWarps * 4 * kPartStride * 4;
  if (red < red_dn) red = red_dn;
  if (red < part) red = part;                                  // the attention's partial states use the same bytes
  const size_t mrg_at = (size_t)kMvWarps * nt_d * 512;         // owners' merge: behind what phase 4 writes there
  if (red < mrg_at + (size_t)16 * kPartStride * 4) red = mrg_at + (size_t)16 * kPartStride * 4;
  L.off_red = (unsigned)o;  o += red;
  L.off_ssq = (unsigned)o;  o += sizeof(float) * kMvWarps * 16;
  L.off_hown = (unsigned)o; o += align_up(sizeof(float) * 16 * (size_t)L.max_nd, 16);
  L.off_zown = (unsigned)o; o += align_up(2 * 16 * (size_t)L.max_nd, 16);
  L.off_mrg = L.off_red + (unsigned)mrg_at;
  o = align_up(o, 128);
  // weights in shared memory as far as they fit, the d-wide ones first
  const size_t wd = (size_t)L.max_nd * L.stride_d * 2, wu = (size_t)L.max_nf * L.stride_d * 2, wn = (size_t)L.max_nd * L.stride_f * 2;
  L.has_d = o + 5 * wd <= max_smem;
  if (L.has_d) { L.off_q = (unsigned)o; L.off_kv = (unsigned)(o + wd); o += 5 * wd; } else { L.off_q = L.off_kv = 0; }
  L.has_up = o + wu <= max_smem;
  L.off_up = L.has_up ? (unsigned)o : 0; if (L.has_up) o += wu;
  L.has_dn = o + wn <= max_smem;
  L.off_dn = L.has_dn ? (unsigned)o : 0; if (L.has_dn) o += wn;
  L.total = (unsigned)o;
  return L;
}

// Exchange area of one layer, in bytes from its start.  Vectors of bf16 are stored as [block of 32 k][16 slots][32 k]: the
// thread (sequence g, quarter c) of an MMA fragment pair reads its eight consecutive k as one 16-byte load.
struct DecWords { size_t c, h, z, g, raw, part, bytes; int seg_max; };

__device__ __forceinline__ float lo_f(unsigned u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float hi_f(unsigned u) { return __uint_as_float(u & 0xffff0000u); }
__device__ __forceinline__ unsigned pack_bf(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const unsigned*>(&v);
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float gelu_erf(float v) { return 0.5f * v * (1.0f + erff(v * 0.70710678118654752f)); }
__device__ __forceinline__ uint4 ld_words(const void* p) {
  unsigned long long a, b;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0,%1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
  return make_uint4((unsigned)a, (unsigned)(a >> 32), (unsigned)b, (unsigned)(b >> 32));
}
__device__ __forceinline__ uint2 ld_words2(const void* p) {
  unsigned long long a;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(a) : "l"(p) : "memory");
  return make_uint2((unsigned)a, (unsigned)(a >> 32));
}
__device__ __forceinline__ void st_word(void* p, unsigned v) { asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory"); }
__device__ __forceinline__ void st_words2(void* p, float a, float b) {
  const unsigned long long w = ((unsigned long long)__float_as_uint(b) << 32) | __float_as_uint(a);
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
// (through the largest of the words: three-input maxima instead of a chain of compares)
__device__ __forceinline__ unsigned top(const uint4& w) { return max(max(max(w.x, w.y), w.z), w.w); }
__device__ __forceinline__ bool full4(const uint4& w) { return top(w) != kEmpty; }
// Fetches 16 bytes again while one of their words is missing.
__device__ __forceinline__ void ld_words_missing(const void* p, uint4& w) {
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %5, 0;\n @q ld.relaxed.gpu.global.v4.u32 {%0,%1,%2,%3}, [%4];\n}"
               : "+r"(w.x), "+r"(w.y), "+r"(w.z), "+r"(w.w) : "l"(p), "r"(full4(w) ? 0u : 1u) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void bulk_prefetch_l2(const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
template <int ID, int N> __device__ __forceinline__ void bar_named() { asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(N) : "memory"); }

// Called every few polls: true when the wait must be given up.  Nobody leaves the kernel early: once a wait has run out
// every later one ends after its first few polls, so all warps reach the end and the status word tells the host.
__device__ __noinline__ bool give_up(SyncArea* s, volatile int* s_abort, unsigned long long* t_start) {
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

// Byte offset of element k of slot b in a vector of the exchange area (16 slots of bf16 or eight of fp32).
template <bool FULL> __device__ __forceinline__ size_t vec_off(int b, int k) {
  return FULL ? ((size_t)((k >> 5) * 8 + b) << 7) + (size_t)(k & 31) * 4 : ((size_t)((k >> 5) * 16 + b) << 6) + (size_t)(k & 31) * 2;
}
// Elements k, k + 1 (k even) into a vector.
template <bool FULL> __device__ __forceinline__ void st_pair(unsigned char* vec, int b, int k, float x0, float x1) {
  if (FULL) st_words2(vec + vec_off<true>(b, k), x0, x1);
  else st_word(vec + vec_off<false>(b, k), pack_bf(x0, x1));
}

// Polls n <= KP blocks of 32 k of a vector (eight consecutive k of slots g and g + 8, or two groups of four of slot g) until every word is
// there; all loads of a round are in flight before any is looked at.  STRIDE: bytes between the two pieces.  (Fetched in place and searched through
// maxima; with copies of what had arrived and a chain of compares a step of 8 layers, B = 16 at 1 k positions, d = 1024, took 375 us instead of 335.)
template <int MB, int KP, int STRIDE>
__device__ __forceinline__ void poll_vec(const unsigned char* base, int n, bool on0, bool on1, uint4 (&a)[KP][MB], SyncArea* sync, volatile int* s_abort) {
#pragma unroll
  for (int i = 0; i < KP; ++i)
#pragma unroll
    for (int r = 0; r < MB; ++r) {
      const unsigned w = i < n && (r ? on1 : on0) ? kEmpty : 0u;
      a[i][r] = make_uint4(w, w, w, w);
    }
  unsigned spins = 0;
  unsigned long long t_start = 0;
  while (true) {
#pragma unroll
    for (int i = 0; i < KP; ++i)
#pragma unroll
      for (int r = 0; r < MB; ++r) ld_words_missing(base + (size_t)i * 1024 + r * STRIDE, a[i][r]);
    unsigned most = 0u;
#pragma unroll
    for (int i = 0; i < KP; ++i)
#pragma unroll
      for (int r = 0; r < MB; ++r) most = max(most, top(a[i][r]));
    if (__all_sync(0xffffffffu, most != kEmpty)) return;
    if ((++spins & 63u) == 0u && __any_sync(0xffffffffu, give_up(sync, s_abort, &t_start))) return;
  }
}
__device__ __forceinline__ uint2 poll2(const void* p, SyncArea* sync, volatile int* s_abort) {
  unsigned spins = 0;
  unsigned long long t_start = 0;
  uint2 w = ld_words2(p);
  while (w.x == kEmpty || w.y == kEmpty) {
    if ((++spins & 63u) == 0u && give_up(sync, s_abort, &t_start)) break;
    w = ld_words2(p);
  }
  return w;
}
__device__ __forceinline__ uint4 poll4(const void* p, SyncArea* sync, volatile int* s_abort) {
  unsigned spins = 0;
  unsigned long long t_start = 0;
  uint4 w = ld_words(p);
  while (!full4(w)) {
    if ((++spins & 63u) == 0u && give_up(sync, s_abort, &t_start)) break;
    w = ld_words(p);
  }
  return w;
}

// A warp's share (n blocks of 32 k) of `tiles` tiles of 8 weight rows; row(t) is this thread's weight row at its first k.
template <int MB, int KP, class RowFn>
__device__ __forceinline__ void tile_products(const uint4 (&a)[KP][MB], int n, int tiles, float4* red, int red_stride, bool add, RowFn row) {
#pragma unroll 1
  for (int t = 0; t < tiles; ++t) {
    const unsigned char* w = row(t);
    float ce[4] = {0.f, 0.f, 0.f, 0.f}, co[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < KP; ++i) {
      const uint4 bw = *reinterpret_cast<const uint4*>(w + (i < n ? i : 0) * 64);      // (blocks beyond n multiply zeros)
      mma16816(ce, a[i][0].x, MB == 2 ? a[i][MB - 1].x : 0u, a[i][0].y, MB == 2 ? a[i][MB - 1].y : 0u, bw.x, bw.y);
      mma16816(co, a[i][0].z, MB == 2 ? a[i][MB - 1].z : 0u, a[i][0].w, MB == 2 ? a[i][MB - 1].w : 0u, bw.z, bw.w);
    }
    float4 v = make_float4(ce[0] + co[0], ce[1] + co[1], ce[2] + co[2], ce[3] + co[3]);
    float4* dst = red + (size_t)t * red_stride;
    if (add) { const float4 o = *dst; v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w; }
    *dst = v;
  }
}
// The same with three terms per value, of up to eight sequences.
template <int KP, class RowFn>
__device__ __forceinline__ void tile_products3(const uint4 (&a)[KP][3], int n, int tiles, float4* red, int red_stride, bool add, RowFn row) {
#pragma unroll 1
  for (int t = 0; t < tiles; ++t) {
    const unsigned char* w = row(t);
    float ce[4] = {0.f, 0.f, 0.f, 0.f}, co[4] = {0.f, 0.f, 0.f, 0.f}, le[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < KP; ++i) {
      const uint4 bw = *reinterpret_cast<const uint4*>(w + (i < n ? i : 0) * 64);      // (blocks beyond n multiply zeros)
      mma16816(ce, a[i][0].x, a[i][1].x, a[i][0].y, a[i][1].y, bw.x, bw.y);
      mma16816(co, a[i][0].z, a[i][1].z, a[i][0].w, a[i][1].w, bw.z, bw.w);
      mma16816(le, a[i][2].x, 0u, a[i][2].y, 0u, bw.x, bw.y);
      mma16816(le, a[i][2].z, 0u, a[i][2].w, 0u, bw.z, bw.w);
    }
    float4 v = make_float4((ce[0] + co[0]) + ((ce[2] + co[2]) + le[0]), (ce[1] + co[1]) + ((ce[3] + co[3]) + le[1]), 0.f, 0.f);
    float4* dst = red + (size_t)t * red_stride;
    if (add) { const float4 o = *dst; v.x += o.x; v.y += o.y; }
    *dst = v;
  }
}
__device__ __forceinline__ float4 sum_parts(const float4* red, int nw) {
  float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
  for (int w = 0; w < nw; ++w) { const float4 v = red[(size_t)w * 32]; y.x += v.x; y.y += v.y; y.z += v.z; y.w += v.w; }
  return y;
}
__device__ __forceinline__ float ssq8(const uint4& w) {
  const float a = lo_f(w.x), b = hi_f(w.x), c = lo_f(w.y), d = hi_f(w.y), e = lo_f(w.z), f = hi_f(w.z), g = lo_f(w.w), h = hi_f(w.w);
  return ((a * a + b * b) + (c * c + d * d)) + ((e * e + f * f) + (g * g + h * h));
}
__device__ __forceinline__ unsigned scale2(unsigned v, unsigned g) { return pack_bf(lo_f(v) * lo_f(g), hi_f(v) * hi_f(g)); }
__device__ __forceinline__ uint4 scale8(const uint4& v, const uint4& g) {
  return make_uint4(scale2(v.x, g.x), scale2(v.y, g.y), scale2(v.z, g.z), scale2(v.w, g.w));
}

// Eight fp32 values (times eight bf16 gains) as three bf16 terms; a value beyond bf16's range keeps its infinity or NaN in the first.
__device__ __forceinline__ void split_pair(float x0, float x1, unsigned& hi, unsigned& mid, unsigned& lo) {
  constexpr float kMax = 3.38e38f;
  hi = pack_bf(x0, x1);
  x0 = fabsf(x0) <= kMax ? x0 - lo_f(hi) : 0.f; x1 = fabsf(x1) <= kMax ? x1 - hi_f(hi) : 0.f;
  mid = pack_bf(x0, x1);
  lo = pack_bf(x0 - lo_f(mid), x1 - hi_f(mid));
}
__device__ __forceinline__ void split8(const uint4& v0, const uint4& v1, const uint4& g, bool scaled, uint4 (&t)[3]) {
  float x[8] = {__uint_as_float(v0.x), __uint_as_float(v0.y), __uint_as_float(v0.z), __uint_as_float(v0.w),
                __uint_as_float(v1.x), __uint_as_float(v1.y), __uint_as_float(v1.z), __uint_as_float(v1.w)};
  if (scaled) {
    x[0] *= lo_f(g.x); x[1] *= hi_f(g.x); x[2] *= lo_f(g.y); x[3] *= hi_f(g.y);
    x[4] *= lo_f(g.z); x[5] *= hi_f(g.z); x[6] *= lo_f(g.w); x[7] *= hi_f(g.w);
  }
  split_pair(x[0], x[1], t[0].x, t[1].x, t[2].x); split_pair(x[2], x[3], t[0].y, t[1].y, t[2].y);
  split_pair(x[4], x[5], t[0].z, t[1].z, t[2].z); split_pair(x[6], x[7], t[0].w, t[1].w, t[2].w);
}
__device__ __forceinline__ float ssq4(const uint4& w) {
  const float a = __uint_as_float(w.x), b = __uint_as_float(w.y), c = __uint_as_float(w.z), d = __uint_as_float(w.w);
  return (a * a + b * b) + (c * c + d * d);
}

template <int MB, bool GAINS, bool FULL>
__global__ void __launch_bounds__(kDecThreads, 1) decode_stack_kernel(const __grid_constant__ DecodeParams p, const DecLayout L, const DecWords W) {
  extern __shared__ __align__(128) unsigned char smem[];
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem);
  float4* red = reinterpret_cast<float4*>(smem + L.off_red);
  float* ssq_red = reinterpret_cast<float*>(smem + L.off_ssq);
  float* hown = reinterpret_cast<float*>(smem + L.off_hown);
  unsigned short* zown = reinterpret_cast<unsigned short*>(smem + L.off_zown);
  float* part_s = reinterpret_cast<float*>(smem + L.off_red);
  float* mrg = reinterpret_cast<float*>(smem + L.off_mrg);
  const uint32_t bar0 = smem_u32(smem + 16);
  const uint32_t bar_q = bar0, bar_kv = bar0 + 8, bar_up = bar0 + 24, bar_dn = bar0 + 32;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x, cta = blockIdx.x, B = p.B, d = p.d, H = p.H, dff = p.dff, n_layers = p.n_layers;
  const int d_lo = 2 * (int)((long long)(d / 2) * cta / G), nd = 2 * (int)((long long)(d / 2) * (cta + 1) / G) - d_lo;
  const int f_lo = 2 * (int)((long long)(dff / 2) * cta / G), nf = 2 * (int)((long long)(dff / 2) * (cta + 1) / G) - f_lo;
  const int nt_d = (nd + 7) / 8, nt_f = (nf + 7) / 8;
  const bool pre = (p.norm_flags & RT_NORM_PRE) != 0, qkn = (p.norm_flags & RT_NORM_QK) != 0;
  const bool kv_norm = pre && !(p.norm_flags & RT_NORM_SKIP_Z);
  const float inv_d = 1.0f / (float)d;
  const int g = lane >> 2, c = lane & 3;
  const bool has0 = g < B, has1 = MB == 2 && g + 8 < B;
  const int pairs = B * H;
  SyncArea* const sync = p.sync;
  static_assert(!FULL || MB == 1, "three terms take the rows of sequences 8 to 15");
  constexpr int KP = FULL ? 2 : 4, NP = FULL ? 2 : MB;         // blocks of 32 k in flight (FULL: two, or the terms would not fit the registers); 16-byte pieces per block and thread
  constexpr int kPiece = FULL ? 16 : 512;                      // bytes between the pieces
  const int vec_at = FULL ? g * 128 + c * 32 : g * 64 + c * 16;

  if (tid == 0) {
    *s_abort = 0;
    for (int i = 0; i < 5; ++i) mbar_init(bar0 + 8 * i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  // ---- weight slices: one warp issues a slice's rows as bulk copies that report to the slice's mbarrier ----
  auto rows_in = [&](uint32_t bar, unsigned off, int stride, const void* Wm, int row_lo, int rows, int K) {
    const unsigned char* src = reinterpret_cast<const unsigned char*>(Wm) + (size_t)row_lo * K * 2;
    for (int r = lane; r < rows; r += 32) bulk_copy(smem_u32(smem + off) + (uint32_t)(r * stride * 2), src + (size_t)r * K * 2, (uint32_t)K * 2u, bar);
  };
  auto expect = [&](uint32_t bar, int rows, int K) {
    if (lane == 0) mbar_expect_tx(bar, (uint32_t)rows * (uint32_t)K * 2u);
    __syncwarp();
  };
  const unsigned wd_bytes = (unsigned)(L.max_nd * L.stride_d * 2);
  auto fetch_q = [&](const void* Wm) { if (L.has_d) { expect(bar_q, nd, d); rows_in(bar_q, L.off_q, L.stride_d, Wm, d_lo, nd, d); } };
  auto fetch_kv = [&](int l) {
    if (!L.has_d) return;
    const uint32_t bar = bar_kv + 8 * (l & 1);
    const unsigned off = L.off_kv + (unsigned)(l & 1) * 2u * wd_bytes;
    expect(bar, 2 * nd, d);
    rows_in(bar, off, L.stride_d, p.layer[l].w_k, d_lo, nd, d);
    rows_in(bar, off + wd_bytes, L.stride_d, p.layer[l].w_v, d_lo, nd, d);
  };
  auto fetch_up = [&](int l) { if (L.has_up) { expect(bar_up, nf, d); rows_in(bar_up, L.off_up, L.stride_d, p.layer[l].w_up, f_lo, nf, d); } };
  auto fetch_dn = [&](int l) { if (L.has_dn) { expect(bar_dn, nd, dff); rows_in(bar_dn, L.off_dn, L.stride_f, p.layer[l].w_down, d_lo, nd, dff); } };
  // start and row stride in bytes of a slice, in shared memory or in place
  auto slice = [&](bool res, unsigned off, int stride, const void* Wm, int row_lo, int K, const unsigned char*& base, size_t& rs) {
    if (res) { base = smem + off; rs = (size_t)stride * 2; }
    else { base = reinterpret_cast<const unsigned char*>(Wm) + (size_t)row_lo * K * 2; rs = (size_t)K * 2; }
  };
  if (warp == kDecWarps - 1) {
    fetch_q(p.layer[0].w_q);
    fetch_kv(0);
    if (n_layers > 1) fetch_kv(1);
    fetch_up(0);
    fetch_dn(0);
  }

  // ---- the attention's split: warp wi takes chunk wi % chunks of the four consecutive (sequence, head) pairs wi / chunks ----
  const int units = p.quads * p.chunks, wpc = p.warps_per_cta;
  const size_t cache_row = (size_t)p.Bs * d, cache_col = (size_t)p.b0 * d;
  // L2 prefetch of (the first part of) the cache rows this CTA's chunks of layer l will read
  auto prefetch_cache = [&](int l) {
    if (p.pf_keys <= 0) return;
    for (int w = warp - kMvWarps; w < wpc; w += kDecWarps - kMvWarps) {
      const int wi = cta * wpc + w;
      if (wi >= units) break;
      const int quad = wi / p.chunks, j0 = (wi % p.chunks) * p.chunk_len;
      const int n = min(min(p.chunk_len, p.pf_keys), p.pos - j0), np = min(4, pairs - quad * 4);
      const size_t col = cache_col + (size_t)quad * 4 * kHeadDim;
      for (int j = lane; j < n; j += 32) {
        const size_t at = (size_t)(j0 + j) * cache_row + col;
        bulk_prefetch_l2(reinterpret_cast<const __nv_bfloat16*>(p.layer[l].k_cache) + at, (uint32_t)np * 128u);
        bulk_prefetch_l2(reinterpret_cast<const __nv_bfloat16*>(p.layer[l].v_cache) + at, (uint32_t)np * 128u);
      }
    }
  };
  if (warp >= kMvWarps) prefetch_cache(0);

  for (int l = 0; l <= n_layers; ++l) {
    const bool last = l == n_layers;                           // only the persistent pair of the last layer is left
    unsigned char* const xw = p.words + (size_t)l * W.bytes;  // exchange area of layer l
    const DecLayer& ly = p.layer[last ? l - 1 : l];
    // =================== 1. projections of x = z^{l-1} (all five matrices in one pass) ===================
    if (warp < kMvWarps) {
      const int nkp = d >> 5, per = (nkp + kMvWarps - 1) / kMvWarps, kp0 = warp * per, kp1 = min(kp0 + per, nkp);
      float sq0 = 0.f, sq1 = 0.f;                              // (FULL: of x, which is z in the storage type, and of z)
      const int m_lo = last ? 3 : 0, m_hi = l == 0 ? 3 : 5;
      if (kp0 >= kp1)
        for (int t = m_lo * nt_d; t < m_hi * nt_d; ++t) red[(t * kMvWarps + warp) * 32 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int k0 = kp0; k0 < kp1; k0 += KP) {
        const int n = min(KP, kp1 - k0);
        uint4 a[KP][MB], zf[FULL ? KP : 1][2], zt[FULL ? KP : 1][3];
        if (l == 0) {
#pragma unroll
          for (int i = 0; i < KP; ++i)
#pragma unroll
            for (int r = 0; r < MB; ++r) {
              a[i][r] = make_uint4(0u, 0u, 0u, 0u);
              const int b = g + 8 * r;
              if (i < n && b < B) {
                const __nv_bfloat16* row;
                if (p.x) row = reinterpret_cast<const __nv_bfloat16*>(p.x) + (size_t)b * p.x_bs;
                else { int id = p.ids[b]; id = id < 0 ? 0 : (id >= p.vocab ? p.vocab - 1 : id); row = reinterpret_cast<const __nv_bfloat16*>(p.emb) + (size_t)id * d; }
                a[i][r] = *reinterpret_cast<const uint4*>(row + (k0 + i) * 32 + 8 * c);
              }
            }
        } else if constexpr (FULL) {
          poll_vec<2, KP, kPiece>(xw - W.bytes + W.z + (size_t)k0 * 1024 + vec_at, n, has0, has0, zf, sync, s_abort);
#pragma unroll
          for (int i = 0; i < KP; ++i) {
            split8(zf[i][0], zf[i][1], zf[i][0], false, zt[i]);
            a[i][0] = zt[i][0];
            sq1 += ssq4(zf[i][0]) + ssq4(zf[i][1]);
          }
        } else {
          poll_vec<MB, KP, kPiece>(xw - W.bytes + W.z + (size_t)k0 * 1024 + vec_at, n, has0, has1, a, sync, s_abort);
        }
#pragma unroll
        for (int i = 0; i < KP; ++i) { sq0 += ssq8(a[i][0]); if (MB == 2) sq1 += ssq8(a[i][MB - 1]); }
        if (k0 == kp0 && L.has_d && !last) {
          mbar_wait(bar_q, 0, s_abort, sync);                  // W_q is always an even fill of its place
          mbar_wait(bar_kv + 8 * (l & 1), (l >> 1) & 1, s_abort, sync);
        }
#pragma unroll 1
        for (int set = 0; set < 2; ++set) {                    // RMS(x) with g_attn for the first three matrices, RMS(z) with g_kv for the others
          if (set == 0 ? last : l == 0) continue;
          uint4 ag[KP][MB];
          const void* gain = set == 0 ? ly.g_attn : p.layer[l - 1].g_kv;
          const bool scaled = GAINS && gain && (set == 0 ? pre : kv_norm);
#pragma unroll
          for (int i = 0; i < KP; ++i) {
            uint4 gv = make_uint4(0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u);
            if (scaled && i < n) gv = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(gain) + (k0 + i) * 32 + 8 * c);
#pragma unroll
            for (int r = 0; r < MB; ++r) ag[i][r] = scaled ? scale8(a[i][r], gv) : a[i][r];
          }
          const int m0 = set == 0 ? 0 : 3, nm = set == 0 ? 3 : 2;
          auto weight_row = [&](int t) {
            const int mt = nt_d == 1 ? t : t / nt_d, m = m0 + mt, r0 = (t - mt * nt_d) * 8, r = r0 + (g < nd - r0 ? g : nd - r0 - 1);
            const unsigned char* base; size_t rs;
            const int lw = m < 3 ? l : l - 1;
            const unsigned kv_off = L.off_kv + (unsigned)(lw & 1) * 2u * wd_bytes;
            if (m == 0) slice(L.has_d, L.off_q, L.stride_d, ly.w_q, d_lo, d, base, rs);
            else if (m == 1 || m == 3) slice(L.has_d, kv_off, L.stride_d, p.layer[lw].w_k, d_lo, d, base, rs);
            else slice(L.has_d, kv_off + wd_bytes, L.stride_d, p.layer[lw].w_v, d_lo, d, base, rs);
            return base + (size_t)r * rs + (size_t)k0 * 64 + c * 16;
          };
          float4* dst = red + ((size_t)m0 * nt_d * kMvWarps + warp) * 32 + lane;
          if constexpr (FULL) {
            if (set == 1) {                                    // the pair comes from z in fp32
              if (scaled) {
#pragma unroll
                for (int i = 0; i < KP; ++i)
                  split8(zf[i][0], zf[i][1], *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(gain) + (k0 + (i < n ? i : 0)) * 32 + 8 * c), true, zt[i]);
              }
              tile_products3<KP>(zt, n, nm * nt_d, dst, kMvWarps * 32, k0 > kp0, weight_row);
              continue;
            }
          }
          tile_products<MB, KP>(ag, n, nm * nt_d, dst, kMvWarps * 32, k0 > kp0, weight_row);
        }
      }
      sq0 += __shfl_xor_sync(0xffffffffu, sq0, 1); sq0 += __shfl_xor_sync(0xffffffffu, sq0, 2);
      sq1 += __shfl_xor_sync(0xffffffffu, sq1, 1); sq1 += __shfl_xor_sync(0xffffffffu, sq1, 2);
      if (c == 0) { ssq_red[warp * 16 + g] = sq0; ssq_red[warp * 16 + 8 + g] = sq1; }
      bar_named<1, kMvWarps * 32>();
      for (int t = m_lo * nt_d + warp; t < m_hi * nt_d; t += kMvWarps) {
        const int m = nt_d == 1 ? t : t / nt_d, rl = (t - m * nt_d) * 8 + 2 * c;
        const float4 y = sum_parts(red + (size_t)t * kMvWarps * 32 + lane, kMvWarps);
        float rs0 = 1.f, rs1 = 1.f;
        if (m < 3 ? pre : kv_norm) {
          float s0 = 0.f, s1 = 0.f;
#pragma unroll
          for (int w = 0; w < kMvWarps; ++w) { s0 += ssq_red[w * 16 + g]; s1 += ssq_red[w * 16 + 8 + g]; }
          rs0 = rsqrtf((FULL && m >= 3 ? s1 : s0) * inv_d + p.eps); rs1 = rsqrtf(s1 * inv_d + p.eps);
        }
        if (rl < nd) {
          unsigned char* dst = xw + W.raw + ((size_t)m * B * d + d_lo + rl) * 4;
          if (has0) st_words2(dst + (size_t)g * d * 4, y.x * rs0, y.y * rs0);
          if (has1) st_words2(dst + (size_t)(g + 8) * d * 4, y.z * rs1, y.w * rs1);
        }
      }
    }
    const int half = warp >> 3, wl = warp & 7;                 // owners' side: two groups of eight warps, a (sequence, head) pair each
    if (!last) {
      // =================== 2. attention over the cache ===================
      const int wi0 = cta * wpc, nw = max(0, min(wpc, units - wi0));
      const bool has_unit = warp < nw;
      float m = -INFINITY, lsum = 0.f, o[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) o[e] = 0.f;
      const int pi = lane >> 3, e0 = 8 * (lane & 7);
      if (has_unit) {
        const int wi = wi0 + warp, quad = wi / p.chunks, j0 = (wi % p.chunks) * p.chunk_len, j1 = min(j0 + p.chunk_len, p.pos);
        const int u = min(quad * 4 + pi, pairs - 1), h = u % H;
        const size_t col = cache_col + (size_t)u * kHeadDim + e0;
        const __nv_bfloat16* kc = reinterpret_cast<const __nv_bfloat16*>(ly.k_cache) + col;
        const __nv_bfloat16* vc = reinterpret_cast<const __nv_bfloat16*>(ly.v_cache) + col;
        const float slope = ly.alibi ? ly.alibi[h] * kLog2e : 0.f;
        float q[8];
        for (int jb = j0; jb < j1; jb += kKeys) {
          uint4 kw[kKeys], vw[kKeys];
#pragma unroll
          for (int i = 0; i < kKeys; ++i) {
            const size_t at = (size_t)min(jb + i, j1 - 1) * cache_row;
            asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(kw[i].x), "=r"(kw[i].y), "=r"(kw[i].z), "=r"(kw[i].w) : "l"(kc + at));
            asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(vw[i].x), "=r"(vw[i].y), "=r"(vw[i].z), "=r"(vw[i].w) : "l"(vc + at));
          }
          if (jb == j0) {                                      // the query arrives while the first rows are on their way
            const unsigned char* qp = xw + W.raw + ((size_t)u * kHeadDim + e0) * 4;
            const uint4 q0 = poll4(qp, sync, s_abort), q1 = poll4(qp + 16, sync, s_abort);
            __syncwarp();
            q[0] = __uint_as_float(q0.x); q[1] = __uint_as_float(q0.y); q[2] = __uint_as_float(q0.z); q[3] = __uint_as_float(q0.w);
            q[4] = __uint_as_float(q1.x); q[5] = __uint_as_float(q1.y); q[6] = __uint_as_float(q1.z); q[7] = __uint_as_float(q1.w);
            float ss = 0.f;
#pragma unroll
            for (int e = 0; e < 8; ++e) ss += q[e] * q[e];
            ss += __shfl_xor_sync(0xffffffffu, ss, 1); ss += __shfl_xor_sync(0xffffffffu, ss, 2); ss += __shfl_xor_sync(0xffffffffu, ss, 4);
            const float rs = qkn ? rsqrtf(ss * (1.0f / kHeadDim) + p.eps) : 1.0f;
#pragma unroll
            for (int e = 0; e < 8; ++e)                        // qkRMS, then the storage rounding
              q[e] = round_T<__nv_bfloat16>(q[e] * rs * (GAINS && qkn ? gain_at(reinterpret_cast<const __nv_bfloat16*>(ly.g_q), h * kHeadDim + e0 + e) : 1.0f));
          }
          float s[kKeys], mx = m;
#pragma unroll
          for (int i = 0; i < kKeys; ++i) {
            float x0 = lo_f(kw[i].x) * q[0], x1 = hi_f(kw[i].x) * q[1];
            x0 = fmaf(lo_f(kw[i].y), q[2], x0); x1 = fmaf(hi_f(kw[i].y), q[3], x1);
            x0 = fmaf(lo_f(kw[i].z), q[4], x0); x1 = fmaf(hi_f(kw[i].z), q[5], x1);
            x0 = fmaf(lo_f(kw[i].w), q[6], x0); x1 = fmaf(hi_f(kw[i].w), q[7], x1);
            s[i] = x0 + x1;
          }
#pragma unroll
          for (int off = 1; off <= 4; off <<= 1)
#pragma unroll
            for (int i = 0; i < kKeys; ++i) s[i] += __shfl_xor_sync(0xffffffffu, s[i], off);
#pragma unroll
          for (int i = 0; i < kKeys; ++i) {
            s[i] = jb + i < j1 ? s[i] * p.scale_log2 - slope * (float)(p.pos - jb - i) : -INFINITY;
            mx = fmaxf(mx, s[i]);
          }
          const float corr = ex2(m - mx);                      // 0 for the first group; mx is finite: the group holds a position
          m = mx;
          lsum *= corr;
#pragma unroll
          for (int e = 0; e < 8; ++e) o[e] *= corr;
#pragma unroll
          for (int i = 0; i < kKeys; ++i) {
            const float w = ex2(s[i] - m);
            lsum += w;
            o[0] = fmaf(w, lo_f(vw[i].x), o[0]); o[1] = fmaf(w, hi_f(vw[i].x), o[1]);
            o[2] = fmaf(w, lo_f(vw[i].y), o[2]); o[3] = fmaf(w, hi_f(vw[i].y), o[3]);
            o[4] = fmaf(w, lo_f(vw[i].z), o[4]); o[5] = fmaf(w, hi_f(vw[i].z), o[5]);
            o[6] = fmaf(w, lo_f(vw[i].w), o[6]); o[7] = fmaf(w, hi_f(vw[i].w), o[7]);
          }
        }
      }
      __syncthreads();                                         // phase 1's partial sums have been read
      if (has_unit) {
        float* dst = part_s + (warp * 4 + pi) * kPartStride;
        *reinterpret_cast<float4*>(dst + e0) = make_float4(o[0], o[1], o[2], o[3]);
        *reinterpret_cast<float4*>(dst + e0 + 4) = make_float4(o[4], o[5], o[6], o[7]);
        if ((lane & 7) == 0) *reinterpret_cast<float2*>(dst + kHeadDim) = make_float2(m, lsum);
      }
      __syncthreads();
      // the places of W_q and of the previous layer's W_k, W_v are free
      if (warp == kDecWarps - 1) { fetch_q(ly.w_o); if (l >= 1 && l + 1 < n_layers) fetch_kv(l + 1); }
      if (nw > 0) {
        // this CTA's warps of one quad become one partial state (256 threads per quad: pair, dimension)
        const int qa = wi0 / p.chunks, qb = (wi0 + nw - 1) / p.chunks, pj = (tid >> 6) & 3, e = tid & 63;
        for (int quad = qa + (tid >> 8); quad <= qb; quad += 2) {
          const int u = quad * 4 + pj;
          if (u >= pairs) continue;
          const int w_lo = max(0, quad * p.chunks - wi0), w_hi = min(nw, (quad + 1) * p.chunks - wi0);
          float M = -INFINITY, so = 0.f, sl = 0.f;
          for (int w = w_lo; w < w_hi; ++w) M = fmaxf(M, part_s[(w * 4 + pj) * kPartStride + kHeadDim]);
          for (int w = w_lo; w < w_hi; ++w) {
            const float* src = part_s + (w * 4 + pj) * kPartStride;
            const float f = ex2(src[kHeadDim] - M);
            so = fmaf(f, src[e], so);
            sl = fmaf(f, src[kHeadDim + 1], sl);
          }
          const int seg = cta - quad * p.chunks / wpc;
          unsigned char* dst = xw + W.part + ((size_t)u * W.seg_max + seg) * kPartStride * 4;
          st_word(dst + e * 4, __float_as_uint(so));
          if (e == 0) st_words2(dst + kHeadDim * 4, M, sl);
        }
      }
      __syncthreads();                                         // the warps' states have been read: mrg may be written
      // =================== 3. owners fold the partial states into the seed of the temporary pair ===================
      for (int k = half; cta + k * G < pairs; k += 2) {
        const int u = cta + k * G, b = u / H, h = u % H, quad = u >> 2;
        float m2 = -INFINITY, l2 = 0.f, o0 = 0.f, o1 = 0.f;
        if (p.chunks > 0) {
          const int first = quad * p.chunks / wpc, nseg = ((quad + 1) * p.chunks - 1) / wpc - first + 1;
          for (int seg = wl; seg < nseg; seg += 8) {
            const unsigned char* src = xw + W.part + ((size_t)u * W.seg_max + seg) * kPartStride * 4;
            const uint2 ow = poll2(src + lane * 8, sync, s_abort), mw = poll2(src + kHeadDim * 4, sync, s_abort);
            __syncwarp();
            const float mc = __uint_as_float(mw.x), mn = fmaxf(m2, mc), f0 = ex2(m2 - mn), f1 = ex2(mc - mn);
            o0 = o0 * f0 + __uint_as_float(ow.x) * f1; o1 = o1 * f0 + __uint_as_float(ow.y) * f1;
            l2 = l2 * f0 + __uint_as_float(mw.y) * f1;
            m2 = mn;
          }
        }
        float* mine = mrg + (half * 8 + wl) * kPartStride;
        *reinterpret_cast<float2*>(mine + 2 * lane) = make_float2(o0, o1);
        if (lane == 0) *reinterpret_cast<float2*>(mine + kHeadDim) = make_float2(m2, l2);
        float sm = 0.f, v0 = 0.f, v1 = 0.f;
        if (wl == 0) {                                         // seed: logit of the temporary pair, l = 1, o = v~
          const unsigned char* src = xw + W.raw + ((size_t)b * d + h * kHeadDim + 2 * lane) * 4;
          const uint2 qw = poll2(src, sync, s_abort), kw = poll2(src + (size_t)B * d * 4, sync, s_abort), vw = poll2(src + (size_t)2 * B * d * 4, sync, s_abort);
          __syncwarp();
          float q0 = __uint_as_float(qw.x), q1 = __uint_as_float(qw.y), k0 = __uint_as_float(kw.x), k1 = __uint_as_float(kw.y);
          if (qkn) {
            const float rq = rsqrtf(warp_sum(q0 * q0 + q1 * q1) * (1.0f / kHeadDim) + p.eps), rk = rsqrtf(warp_sum(k0 * k0 + k1 * k1) * (1.0f / kHeadDim) + p.eps);
            const int at = h * kHeadDim + 2 * lane;
            const __nv_bfloat16 *gq = reinterpret_cast<const __nv_bfloat16*>(ly.g_q), *gk = reinterpret_cast<const __nv_bfloat16*>(ly.g_k);
            q0 *= rq * (GAINS ? gain_at(gq, at) : 1.f); q1 *= rq * (GAINS ? gain_at(gq, at + 1) : 1.f);
            k0 *= rk * (GAINS ? gain_at(gk, at) : 1.f); k1 *= rk * (GAINS ? gain_at(gk, at + 1) : 1.f);
          }
          const unsigned qr = pack_bf(q0, q1), kr = pack_bf(k0, k1), vr = pack_bf(__uint_as_float(vw.x), __uint_as_float(vw.y));
          sm = warp_sum(lo_f(qr) * lo_f(kr) + hi_f(qr) * hi_f(kr)) * p.scale_log2;
          v0 = lo_f(vr); v1 = hi_f(vr);
        }
        asm volatile("bar.sync %0, 256;" ::"r"(2 + half) : "memory");
        if (wl == 0) {
          float M = sm;
#pragma unroll
          for (int w = 0; w < 8; ++w) M = fmaxf(M, mrg[(half * 8 + w) * kPartStride + kHeadDim]);
          const float fs = ex2(sm - M);
          float den = fs, a0 = v0 * fs, a1 = v1 * fs;
#pragma unroll
          for (int w = 0; w < 8; ++w) {
            const float* src = mrg + (half * 8 + w) * kPartStride;
            const float f = ex2(src[kHeadDim] - M);            // 0 for a warp without a partial state
            const float2 ow = *reinterpret_cast<const float2*>(src + 2 * lane);
            a0 = fmaf(f, ow.x, a0); a1 = fmaf(f, ow.y, a1); den = fmaf(f, src[kHeadDim + 1], den);
          }
          const float inv = 1.0f / den;
          st_pair<FULL>(xw + W.c, b, h * kHeadDim + 2 * lane, a0 * inv, a1 * inv);
        }
        if (cta + (k + 2) * G < pairs) asm volatile("bar.sync %0, 256;" ::"r"(2 + half) : "memory");
      }
    }
    if (l > 0 && warp >= kMvWarps) {
      // persistent pair of layer l-1 (Eqs. 1-2): qkRMS of k, cache rows
      const DecLayer& lp = p.layer[l - 1];
      for (int u = cta + (warp - kMvWarps) * G; u < pairs; u += (kDecWarps - kMvWarps) * G) {
        const int b = u / H, at = (u % H) * kHeadDim + 2 * lane;
        const unsigned char* src = xw + W.raw + ((size_t)3 * B * d + (size_t)b * d + at) * 4;
        const uint2 kw = poll2(src, sync, s_abort), vw = poll2(src + (size_t)B * d * 4, sync, s_abort);
        __syncwarp();
        const float k0 = __uint_as_float(kw.x), k1 = __uint_as_float(kw.y);
        const float rk = qkn ? rsqrtf(warp_sum(k0 * k0 + k1 * k1) * (1.0f / kHeadDim) + p.eps) : 1.0f;
        const __nv_bfloat16* gk = reinterpret_cast<const __nv_bfloat16*>(lp.g_k);
        const size_t row = (size_t)p.pos * cache_row + cache_col + (size_t)b * d + at;
        *reinterpret_cast<unsigned*>(reinterpret_cast<__nv_bfloat16*>(lp.k_cache) + row) =
            pack_bf(k0 * rk * (GAINS && qkn ? gain_at(gk, at) : 1.f), k1 * rk * (GAINS && qkn ? gain_at(gk, at + 1) : 1.f));
        *reinterpret_cast<unsigned*>(reinterpret_cast<__nv_bfloat16*>(lp.v_cache) + row) = pack_bf(__uint_as_float(vw.x), __uint_as_float(vw.y));
      }
    }
    if (last) break;
    if (warp >= kMvWarps) {
      // idle until phase 6: ask L2 for what comes next
      if (l + 1 < n_layers) prefetch_cache(l + 1);
      else if (p.next_bytes) {
        const size_t per = (p.next_size / G + 15) & ~(size_t)15, lo = per * cta, hi = lo + per < p.next_size ? lo + per : p.next_size;
        for (size_t at = lo + (size_t)((warp - kMvWarps) * 32 + lane) * 2048; at < hi; at += (size_t)(kDecWarps - kMvWarps) * 32 * 2048)
          bulk_prefetch_l2(reinterpret_cast<const unsigned char*>(p.next_bytes) + at, (uint32_t)((hi - at < 2048 ? hi - at : 2048) & ~(size_t)15));
      }
    } else {
      const int nkp = d >> 5, per = (nkp + kMvWarps - 1) / kMvWarps, kp0 = warp * per, kp1 = min(kp0 + per, nkp);
#pragma unroll 1
      for (int ph = 4; ph <= 5; ++ph) {
        // =================== 4. h = x + alpha W_o c     5. g = GELU(W_up RMS(h)) ===================
        const int rows = ph == 4 ? nd : nf, tiles = ph == 4 ? nt_d : nt_f;
        const unsigned char* base; size_t rs;
        if (ph == 4) slice(L.has_d, L.off_q, L.stride_d, ly.w_o, d_lo, d, base, rs);
        else slice(L.has_up, L.off_up, L.stride_d, ly.w_up, f_lo, d, base, rs);
        float sq0 = 0.f, sq1 = 0.f;
        if (kp0 >= kp1)
          for (int t = 0; t < tiles; ++t) red[(t * kMvWarps + warp) * 32 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k0 = kp0; k0 < kp1; k0 += KP) {
          const int n = min(KP, kp1 - k0);
          uint4 a[KP][NP], at[FULL ? KP : 1][3];
          poll_vec<NP, KP, kPiece>(xw + (ph == 4 ? W.c : W.h) + (size_t)k0 * 1024 + vec_at, n, has0, FULL ? has0 : has1, a, sync, s_abort);
          if constexpr (FULL) {
            const bool scaled = GAINS && ph == 5 && pre && ly.g_mlp;
#pragma unroll
            for (int i = 0; i < KP; ++i) {
              uint4 gv = make_uint4(0u, 0u, 0u, 0u);
              if (scaled) gv = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(ly.g_mlp) + (k0 + (i < n ? i : 0)) * 32 + 8 * c);
              split8(a[i][0], a[i][1], gv, scaled, at[i]);
              sq0 += ssq4(a[i][0]) + ssq4(a[i][1]);
            }
          } else if (ph == 5) {
#pragma unroll
            for (int i = 0; i < KP; ++i) { sq0 += ssq8(a[i][0]); if (MB == 2) sq1 += ssq8(a[i][MB - 1]); }
            if (GAINS && pre && ly.g_mlp) {
#pragma unroll
              for (int i = 0; i < KP; ++i) {
                const uint4 gv = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(ly.g_mlp) + (k0 + (i < n ? i : 0)) * 32 + 8 * c);
#pragma unroll
                for (int r = 0; r < MB; ++r) a[i][r] = scale8(a[i][r], gv);
              }
            }
          }
          if (k0 == kp0) {
            if (ph == 4) { if (L.has_d) mbar_wait(bar_q, 1, s_abort, sync); }
            else if (L.has_up) mbar_wait(bar_up, l & 1, s_abort, sync);
          }
          auto weight_row = [&](int t) {
            const int r0 = t * 8, r = r0 + (g < rows - r0 ? g : rows - r0 - 1);
            return base + (size_t)r * rs + (size_t)k0 * 64 + c * 16;
          };
          if constexpr (FULL) tile_products3<KP>(at, n, tiles, red + warp * 32 + lane, kMvWarps * 32, k0 > kp0, weight_row);
          else tile_products<MB, KP>(a, n, tiles, red + warp * 32 + lane, kMvWarps * 32, k0 > kp0, weight_row);
        }
        if (ph == 5) {
          sq0 += __shfl_xor_sync(0xffffffffu, sq0, 1); sq0 += __shfl_xor_sync(0xffffffffu, sq0, 2);
          sq1 += __shfl_xor_sync(0xffffffffu, sq1, 1); sq1 += __shfl_xor_sync(0xffffffffu, sq1, 2);
          if (c == 0) { ssq_red[warp * 16 + g] = sq0; ssq_red[warp * 16 + 8 + g] = sq1; }
        }
        bar_named<1, kMvWarps * 32>();
        for (int t = warp; t < tiles; t += kMvWarps) {
          const int rl = t * 8 + 2 * c;
          const float4 y = sum_parts(red + (size_t)t * kMvWarps * 32 + lane, kMvWarps);
          if (rl >= rows) continue;
          if (ph == 4) {
#pragma unroll
            for (int r = 0; r < MB; ++r) {
              const int b = g + 8 * r;
              if (b >= B) continue;
              unsigned xv;
              if (l > 0) xv = *reinterpret_cast<const unsigned*>(zown + b * L.max_nd + rl);
              else {
                const __nv_bfloat16* row;
                if (p.x) row = reinterpret_cast<const __nv_bfloat16*>(p.x) + (size_t)b * p.x_bs;
                else { int id = p.ids[b]; id = id < 0 ? 0 : (id >= p.vocab ? p.vocab - 1 : id); row = reinterpret_cast<const __nv_bfloat16*>(p.emb) + (size_t)id * d; }
                xv = *reinterpret_cast<const unsigned*>(row + d_lo + rl);
              }
              const float h0 = lo_f(xv) + p.alpha * (r ? y.z : y.x), h1 = hi_f(xv) + p.alpha * (r ? y.w : y.y);
              *reinterpret_cast<float2*>(hown + b * L.max_nd + rl) = make_float2(h0, h1);
              st_pair<FULL>(xw + W.h, b, d_lo + rl, h0, h1);
            }
          } else {
            float rs0 = 1.f, rs1 = 1.f;
            if (pre) {
              float s0 = 0.f, s1 = 0.f;
#pragma unroll
              for (int w = 0; w < kMvWarps; ++w) { s0 += ssq_red[w * 16 + g]; s1 += ssq_red[w * 16 + 8 + g]; }
              rs0 = rsqrtf(s0 * inv_d + p.eps); rs1 = rsqrtf(s1 * inv_d + p.eps);
            }
            if (has0) st_pair<FULL>(xw + W.g, g, f_lo + rl, gelu_erf(y.x * rs0), gelu_erf(y.y * rs0));
            if (has1) st_pair<FULL>(xw + W.g, g + 8, f_lo + rl, gelu_erf(y.z * rs1), gelu_erf(y.w * rs1));
          }
        }
        bar_named<1, kMvWarps * 32>();                         // red may be written again; the slice's place is free
        if (warp == kMvWarps - 1 && l + 1 < n_layers) { if (ph == 4) fetch_q(p.layer[l + 1].w_q); else fetch_up(l + 1); }
      }
    }
    __syncthreads();                                           // phase 5's sums have been read
    {
      // =================== 6. z = h + alpha W_down g, all sixteen warps ===================
      const int nkp = dff >> 5, per = (nkp + kDecWarps - 1) / kDecWarps, kp0 = warp * per, kp1 = min(kp0 + per, nkp);
      const unsigned char* base; size_t rs;
      slice(L.has_dn, L.off_dn, L.stride_f, ly.w_down, d_lo, dff, base, rs);
      if (kp0 >= kp1)
        for (int t = 0; t < nt_d; ++t) red[(t * kDecWarps + warp) * 32 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int k0 = kp0; k0 < kp1; k0 += KP) {
        const int n = min(KP, kp1 - k0);
        uint4 a[KP][NP], at[FULL ? KP : 1][3];
        poll_vec<NP, KP, kPiece>(xw + W.g + (size_t)k0 * 1024 + vec_at, n, has0, FULL ? has0 : has1, a, sync, s_abort);
        if (k0 == kp0 && L.has_dn) mbar_wait(bar_dn, l & 1, s_abort, sync);
        auto weight_row = [&](int t) {
          const int r0 = t * 8, r = r0 + (g < nd - r0 ? g : nd - r0 - 1);
          return base + (size_t)r * rs + (size_t)k0 * 64 + c * 16;
        };
        if constexpr (FULL) {
#pragma unroll
          for (int i = 0; i < KP; ++i) split8(a[i][0], a[i][1], a[i][0], false, at[i]);
          tile_products3<KP>(at, n, nt_d, red + warp * 32 + lane, kDecWarps * 32, k0 > kp0, weight_row);
        } else tile_products<MB, KP>(a, n, nt_d, red + warp * 32 + lane, kDecWarps * 32, k0 > kp0, weight_row);
      }
      __syncthreads();
      if (warp == kDecWarps - 1 && l + 1 < n_layers) fetch_dn(l + 1);
      if (warp < kMvWarps) {
        for (int t = warp; t < nt_d; t += kMvWarps) {
          const int rl = t * 8 + 2 * c;
          const float4 y = sum_parts(red + (size_t)t * kDecWarps * 32 + lane, kDecWarps);
          if (rl >= nd) continue;
#pragma unroll
          for (int r = 0; r < MB; ++r) {
            const int b = g + 8 * r;
            if (b >= B) continue;
            const float2 h = *reinterpret_cast<const float2*>(hown + b * L.max_nd + rl);
            const float z0 = h.x + p.alpha * (r ? y.z : y.x), z1 = h.y + p.alpha * (r ? y.w : y.y);
            const unsigned zw = pack_bf(z0, z1);
            st_pair<FULL>(xw + W.z, b, d_lo + rl, z0, z1);
            *reinterpret_cast<unsigned*>(zown + b * L.max_nd + rl) = zw;
            if (l == n_layers - 1)
              *reinterpret_cast<unsigned*>(reinterpret_cast<__nv_bfloat16*>(p.z_out) + (size_t)b * p.z_bs + d_lo + rl) = zw;
          }
        }
        bar_named<1, kMvWarps * 32>();                         // red may be written again
      }
    }
  }
  // nobody leaves with a copy in flight (only an aborted run can still have one here)
  if (tid == 0 && *s_abort) {
    for (int i = 0; i < 5; ++i)
      for (int spins = 0; spins < (1 << 16); ++spins) mbar_try_wait(bar0 + 8 * i, 0);
  }
  __syncthreads();
}

DecWords dec_words(int B, int d, int H, int dff, int seg_max) {
  DecWords W;
  size_t o = 0;
  auto take = [&](size_t n) { const size_t at = o; o += align_up(n, 256); return at; };
  W.c = take((size_t)16 * d * 2); W.h = take((size_t)16 * d * 2); W.z = take((size_t)16 * d * 2); W.g = take((size_t)16 * dff * 2);
  W.raw = take((size_t)5 * B * d * 4);
  W.seg_max = seg_max;
  W.part = take((size_t)B * H * seg_max * kPartStride * 4);
  W.bytes = o;
  return W;
}

struct DecDevice { int sms; size_t smem; };
bool dec_device(DecDevice* out) {
  thread_local int dev_cached = -1;
  thread_local DecDevice c;
  int dev = 0, sms = 0, smem = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  if (dev != dev_cached) {
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return false;
    c.sms = sms; c.smem = (size_t)smem;
    dev_cached = dev;
  }
  *out = c;
  return true;
}

// Most partial states per (sequence, head): every CTA that holds a chunk of its four pairs leaves one.
int seg_bound(int quads, int grid) { return ceil_div(grid, quads) + 2; }

}  // namespace

int decode_slice(int B, bool full) { return ceil_div(B, ceil_div(B, full ? 8 : 16)); }

// Widths in whole 64-byte blocks whose reduction buffers leave room in shared memory (five d-wide matrices at once: d up to about 12000 with
// d_ff = 4 d; d_ff up to about 65000), and no more groups of four pairs than warps (pure arithmetic).
bool decode_shape(int B, int d, int H, int dff) {
  return d % 64 == 0 && dff % 32 == 0 && dec_layout(d, dff, kB200Sms, kB200SmemPerCta).total <= kB200SmemPerCta &&
         (long long)(B < 16 ? B : 16) * H <= 4LL * kB200Sms * kDecWarps;
}

// Room for every slice of up to min(B, 16) sequences.  What a slice needs does not grow with it: fewer sequences have fewer groups of four
// pairs, hence more partial states for each pair (d = 128, H = 2: eight sequences need 10 KB a layer more than nine).
size_t decode_words_bytes(int n_layers, int B, int d, int H, int dff) {
  if (B < 1 || !decode_shape(1, d, H, dff)) return 0;
  const int n = n_layers < kDecMaxLayers ? n_layers : kDecMaxLayers;
  size_t most = 0;
  for (int b = 1; b <= B && b <= 16; ++b) {
    const size_t bytes = dec_words(b, d, H, dff, seg_bound(ceil_div(b * H, 4), kB200Sms)).bytes;
    if (bytes > most) most = bytes;
  }
  return (size_t)(n + 1) * most;
}

cudaError_t decode_launch(const DecodeParams& p0, cudaStream_t s) {
  DecodeParams p = p0;
  DecDevice dv;
  if (!dec_device(&dv)) return cudaErrorUnknown;
  const int grid = dv.sms < kB200Sms ? dv.sms : kB200Sms;
  const DecLayout L = dec_layout(p.d, p.dff, grid, dv.smem);
  if (L.total > dv.smem) return cudaErrorInvalidConfiguration;
  // Attention: about one chunk per warp of the grid, at least eight positions each; the chunks of four pairs are
  // consecutive warps, dealt out so that every CTA gets the same number.
  const int pairs = p.B * p.H;
  p.quads = ceil_div(pairs, 4);
  p.chunks = 0; p.chunk_len = kKeys; p.warps_per_cta = 1; p.pf_keys = 0;
  const int seg_max = seg_bound(p.quads, kB200Sms);
  if (p.pos > 0) {
    int want = grid * kDecWarps / p.quads;
    if (want < 1) want = 1;
    p.chunk_len = ceil_div(p.pos, want);
    if (p.chunk_len < kKeys) p.chunk_len = kKeys;
    p.chunks = ceil_div(p.pos, p.chunk_len);
    p.warps_per_cta = ceil_div(p.quads * p.chunks, grid);
    if (p.warps_per_cta > kDecWarps) return cudaErrorInvalidConfiguration;
    // what HBM delivers while the mat-vec phases of a layer run (about 6 us), and no more than a part of L2 holds
    const size_t per_key = (size_t)pairs * 128 * 2 * p.chunks;
    const size_t keys = (size_t)(40u << 20) / per_key;
    p.pf_keys = (int)(keys < (size_t)p.chunk_len ? keys : (size_t)p.chunk_len);
  }
  const DecWords W = dec_words(p.B, p.d, p.H, p.dff, seg_max);
  if ((size_t)(p.n_layers + 1) * W.bytes > p.words_size) return cudaErrorInvalidConfiguration;
  bool gains = false;
  for (int l = 0; l < p.n_layers; ++l)
    gains = gains || p.layer[l].g_attn || p.layer[l].g_mlp || p.layer[l].g_kv || p.layer[l].g_q || p.layer[l].g_k;
  if (p.B > (p.full ? 8 : 16)) return cudaErrorInvalidConfiguration;
  const void* fn = p.full ? (gains ? (const void*)&decode_stack_kernel<1, true, true> : (const void*)&decode_stack_kernel<1, false, true>)
                   : p.B > 8 ? (gains ? (const void*)&decode_stack_kernel<2, true, false> : (const void*)&decode_stack_kernel<2, false, false>)
                             : (gains ? (const void*)&decode_stack_kernel<1, true, false> : (const void*)&decode_stack_kernel<1, false, false>);
  cudaError_t e = ensure_dynamic_smem(fn, (int)L.total);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(p.words, 0xff, (size_t)(p.n_layers + 1) * W.bytes, s);
  if (e != cudaSuccess) return e;
  DecLayout Lc = L;
  DecWords Wc = W;
  void* args[] = {(void*)&p, (void*)&Lc, (void*)&Wc};
  return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kDecThreads), args, L.total, s);
}

}  // namespace rt
