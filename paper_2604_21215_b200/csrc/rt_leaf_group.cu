// Leaf recurrence of several independent (layer, slice of sequences) jobs at once, bf16: the SMs are split into groups of
// equal size, one job each.  Used where jobs exist side by side: the layers of a stack (layer l works on a leaf that layer
// l-1 finished in an earlier launch) and batches of more than 16 sequences (slices of at most 16).
//
// A token step is a chain of exchanges whose length does not depend on how many SMs take part, so a single job leaves
// 148 SMs waiting most of the time (rt_leaf_mma.cu).  Several jobs side by side fill the waits.  A group's weights (23 MB at
// d = 1024) do not stay on chip: every step streams them from L2 through a ring of bulk copies that keeps filling while the
// chain waits.  One SM takes 145 GB/s from L2 (all together 18 TB/s as long as the jobs' weights fit L2), but only in large pieces: a copy costs
// the copy unit about 90 ns whatever its size.  So the weights are packed once per call, in the order in which a CTA uses them.
//
// Exchanges: c, h, g and z travel as packed bf16 in the order the fragments are read; a word that has not been written is all ones, a pair no
// result is (NaN results are 0x7fff), so the words are their own flags and nobody waits for a barrier.  Every vector has four arrays, used by
// turns: the CTA that publishes a word sets it back well before it is used again, once it knows from what it has received since that
// every CTA has read it (see "set back" below).  Raw k|v travel as fp32 words beside their step number (one reader each).
//
// Products are those of rt_leaf_mma.cu, to the bit: m16n8k16 MMAs with the sequences as rows, K split over the eight MMA warps in the same parts,
// the same order of sums, so that layers side by side give the results of the same layers one after the other.  What differs: the weights come by pieces
// of 16 rows, of which the next one is fetched from the ring while the products of the present one run; a phase's activations are fetched once for all its
// pieces; the attention warps own up to three (sequence, head) pairs each and hold nothing of the leaf but the one query that is finished
// next: its earlier pairs are read back from the caches while the mat-vecs run.
//
// What bounds a step (37 SMs a group, d = 1024, B = 16: 45 thousand cycles, clock stamps): a fifth each products (an m16n8k16 takes a scheduler 16 cycles) and waiting for
// words, the rest instructions that run once or a few times per phase: row sums and epilogues 5, partial sums 4, weights not there yet 5, set-up of the phases
// 7 thousand.  Stalls at B = 40, d = 768 (ncu, warps per issue slot): words polled 3.2, fixed latencies 1.9, fences 0.5, instruction fetch 0.4, tensor pipe 0.2.
// Dividing by H in the attention warps and a second copy of their loop (12 KB of code) cost 5 to 15 %.  Measured against the form before
// (counter barrier for g, words with their own step number, windows of 16 queries, four places): 8 layers of d = 1024, B = 16, N = 2048 220 (one by one) -> 114 ms;
// B = 1, N = 77 4.77 -> 4.41; 8 layers of d = 768, B = 16, N = 512 31.9 -> 20.4; one layer, B = 40, d = 768, N = 333 7.0 -> 5.5, B = 64, d = 1024 9.65 -> 7.0.
// Tried: warps of their own for the row sums (640 threads, 152 registers: slower, 36 against 31 ms for B = 16, N = 512); polling one word before the rest and
// the attention warps asleep until this CTA has z (3 % slower); pieces double-buffered in registers with a barrier per chunk (4 % slower).
#include <cuda_bf16.h>
#include <string.h>

#include <type_traits>

#include "rt_kernels.h"
#include "rt_tc.cuh"

namespace rt {

namespace {

constexpr int kGMma = 8, kGAtt = 7;               // MMA warps, attention warps; the last warp issues the copies
constexpr int kGThreads = (kGMma + kGAtt + 1) * 32;
constexpr int kGRegsMma = 184, kGRegsRest = 72;   // (184 + 72) * 256 = 65536
constexpr int kTurns = 4;                         // arrays of each exchanged vector, used by turns
constexpr int kQuad = 2 * 2;                      // tiles a warp works on at a time: two pieces
constexpr int kMaxSlots = 16;
constexpr int kKP = 4;                            // blocks of 32 k per warp and stretch
constexpr int kPieceTiles = 2;                    // tiles of 8 weight rows per piece
constexpr int kMaxPairs = 3;                      // (sequence, head) pairs per attention warp
constexpr int kFoldKeys = 8, kFoldLanes = 32 / kFoldKeys;      // earlier pairs of the leaf absorbed at a time

// How a group of g CTAs shares the rows; a CTA's pieces of a step in order: W_o, W_up, W_down (stretch by stretch), W_k | W_v.
// max_nd, max_nf, nt_d, nt_f: upper bounds over the CTAs.  The contraction is cut into blocks of 32 k; a warp has bd consecutive ones of d, bf of
// d_ff, the latter in nq stretches of at most kKP.
struct GroupShape { int max_nd, max_nf, nt_d, nt_f, bd, bf, nq; uint32_t tile_d, step_bytes; };
__host__ __device__ inline GroupShape group_shape(int d, int dff, int g) {
  GroupShape s;
  s.max_nd = 2 * ((d / 2 + g - 1) / g);
  s.max_nf = 2 * ((dff / 2 + g - 1) / g);
  s.nt_d = (s.max_nd + 7) / 8; s.nt_f = (s.max_nf + 7) / 8;
  s.bd = (d / 32 + kGMma - 1) / kGMma;
  s.bf = (dff / 32 + kGMma - 1) / kGMma;
  s.nq = (s.bf + kKP - 1) / kKP;
  s.tile_d = (uint32_t)(16 * d);                  // [d / 32][8 rows][32]: the 16-byte fragment loads of eight lanes cover 128 bytes
  s.step_bytes = (uint32_t)(3 * s.nt_d + s.nt_f) * s.tile_d + (uint32_t)(s.nt_d * s.bf * kGMma * 512);
  return s;
}
// Blocks per warp in stretch q of W_down; a tile of the stretch is [8 warps][blocks][8 rows][32].
__host__ __device__ inline int stretch_blocks(const GroupShape& s, int q) { const int left = s.bf - kKP * q; return left < kKP ? left : kKP; }

struct GroupLayout {
  int slots;                                      // ring entries
  GroupShape s;
  uint32_t off_red, off_ssq, off_ring, slot_bytes, total;
};

GroupLayout group_layout(int d, int dff, int g, size_t max_smem) {
  GroupLayout L;
  L.s = group_shape(d, dff, g);
  uint32_t o = 512;
  auto take = [&](uint32_t n) { o = (o + 127) / 128 * 128; const uint32_t at = o; o += n; return at; };
  L.off_red = take(2 * kGMma * kGMma * 32 * 8);   // two buffers of eight (tile, half of the sequences) units
  L.off_ssq = take(kGMma * 16 * 4);
  L.off_ring = (o + 127) / 128 * 128;
  const uint32_t tile_f = (uint32_t)(kGMma * stretch_blocks(L.s, 0) * 512);
  L.slot_bytes = kPieceTiles * (L.s.tile_d > tile_f ? L.s.tile_d : tile_f);
  L.slots = max_smem > L.off_ring ? (int)((max_smem - L.off_ring) / L.slot_bytes) : 0;
  if (L.slots > kMaxSlots) L.slots = kMaxSlots;
  L.total = L.off_ring + (uint32_t)L.slots * L.slot_bytes;
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
constexpr unsigned kUnset = 0xffffffffu;
__device__ __forceinline__ unsigned top(const uint4& w) { return max(max(max(w.x, w.y), w.z), w.w); }
__device__ __forceinline__ bool unset(const uint4& w) { return top(w) == kUnset; }
// Fetches 16 bytes again while one of their words has not been written.
__device__ __forceinline__ void ld_unset(const void* p, uint4& w) {
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %5, 0;\n @q ld.relaxed.gpu.global.v4.u32 {%0,%1,%2,%3}, [%4];\n}"
               : "+r"(w.x), "+r"(w.y), "+r"(w.z), "+r"(w.w) : "l"(p), "r"(unset(w) ? 1u : 0u) : "memory");
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ void st_word(void* p, unsigned v) { asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory"); }
__device__ __forceinline__ void st_flag2(void* p, unsigned a, unsigned b, unsigned seq) {
  const unsigned long long w0 = ((unsigned long long)seq << 32) | a, w1 = ((unsigned long long)seq << 32) | b;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1,%2};" ::"l"(p), "l"(w0), "l"(w1) : "memory");
}
__device__ __forceinline__ void gmma(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ bool group_give_up(SyncArea* s, volatile int* s_abort, unsigned long long* t_start) {
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
// Waits for an mbarrier of this CTA; false when the wait was given up.
__device__ __forceinline__ bool ring_wait_slow(uint32_t bar, uint32_t parity, SyncArea* s, volatile int* s_abort) {
  unsigned spins = 0;
  unsigned long long t0 = 0;
  while (!mbar_try_wait(bar, parity))
    if ((++spins & 255u) == 0u && group_give_up(s, s_abort, &t0)) return false;
  return true;
}
__device__ __forceinline__ bool ring_wait(uint32_t bar, uint32_t parity, SyncArea* s, volatile int* s_abort) {
  return mbar_try_wait(bar, parity) || ring_wait_slow(bar, parity, s, s_abort);
}
// Where element k lies in a block of 32 k of an exchanged vector or a packed weight row: a thread's sixteen bytes are the four elements that it
// feeds to the products of the block's first 16 k, then the four of the second.
__host__ __device__ __forceinline__ int in_block(int k) { return ((k & 15) >> 2) * 8 + ((k >> 4) & 1) * 4 + (k & 3); }
// Byte offset of elements k, k + 1 (k even) of slot b of an exchanged vector: [block of 32 k][16 slots][32 k].
__device__ __forceinline__ uint32_t w_off(int b, int k) { return ((uint32_t)((k >> 5) * 16 + b) << 6) + (uint32_t)in_block(k) * 2; }

struct GroupArgs {
  GroupCommon c;
  GroupJob job[kGroupJobs];
  int n_jobs, gsize;
};

// Packs one layer: a CTA's tiles one after the other in the order of use, rows and blocks beyond its own zero.
__global__ void __launch_bounds__(256) group_pack_kernel(const __grid_constant__ GroupPackArgs a) {
  const GroupShape s = group_shape(a.d, a.dff, a.g);
  const int cta = blockIdx.x, layer = blockIdx.z;
  const GroupPackLayer& w = a.layer[layer];
  const int d_lo = 2 * (int)((long long)(a.d / 2) * cta / a.g), nd = 2 * (int)((long long)(a.d / 2) * (cta + 1) / a.g) - d_lo;
  const int f_lo = 2 * (int)((long long)(a.dff / 2) * cta / a.g), nf = 2 * (int)((long long)(a.dff / 2) * (cta + 1) / a.g) - f_lo;
  int t = blockIdx.y, rows = nd, row = d_lo, K = a.d, q = -1, nb = s.bd;
  uint32_t at = 0;                                             // where the tile begins
  const void* src;
  if (t < s.nt_d) { src = w.w_o; at = t * s.tile_d; }
  else if ((t -= s.nt_d) < s.nt_f) { src = w.w_up; rows = nf; row = f_lo; at = (s.nt_d + t) * s.tile_d; }
  else if ((t -= s.nt_f) < s.nt_d * s.nq) {
    src = w.w_down; K = a.dff; q = t / s.nt_d; t %= s.nt_d; nb = stretch_blocks(s, q);
    at = (s.nt_d + s.nt_f) * s.tile_d + (uint32_t)(s.nt_d * q * kKP * kGMma * 512) + (uint32_t)(t * nb * kGMma * 512);
  } else {
    t -= s.nt_d * s.nq;
    at = (s.nt_d + s.nt_f + t) * s.tile_d + (uint32_t)(s.nt_d * s.bf * kGMma * 512);
    src = t < s.nt_d ? w.w_k : w.w_v;
    t %= s.nt_d;
  }
  const int n_blocks = q < 0 ? a.d / 32 : kGMma * nb;          // blocks of 8 rows x 32 k: 64 threads copy 8 bytes each
  unsigned char* dst = reinterpret_cast<unsigned char*>(w.out) + (size_t)cta * s.step_bytes + at;
  const int r = (threadIdx.x & 63) >> 3, k4 = (threadIdx.x & 7) * 4;      // consecutive threads read consecutive 8-byte groups of a row
  for (int blk = threadIdx.x >> 6; blk < n_blocks; blk += 4) {
    // first k of the block, and whether the warp that multiplies by it has it
    const int i = q < 0 ? blk : (blk / nb) * s.bf + q * kKP + blk % nb, k = i * 32 + k4;
    uint2 v = make_uint2(0u, 0u);
    if (t * 8 + r < rows && k < K) v = *reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(src) + (size_t)(row + t * 8 + r) * K + k);
    *reinterpret_cast<uint2*>(dst + blk * 512 + r * 64 + in_block(k4) * 2) = v;
  }
}

// PW: (sequence, head) pairs per attention warp.
template <int MB, int PW>
__global__ void __launch_bounds__(kGThreads, 1) leaf_group_kernel(const __grid_constant__ GroupArgs a, const __grid_constant__ GroupLayout L) {
  extern __shared__ __align__(128) unsigned char smem[];
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem);
  const uint32_t full = smem_u32(smem + 64), empty = full + 8 * kMaxSlots, red_full = empty + 8 * kMaxSlots, cleared = red_full + 16;
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
  // exchange area: c, h, z, g once per turn, then raw k|v
  const uint32_t vec = (uint32_t)(32 * d), set = 3 * vec + (uint32_t)(32 * dff);
  unsigned char *const words = J.words, *const w_kv = words + kTurns * (size_t)set;
  auto c_of = [&](unsigned step) { return words + (size_t)(step % kTurns) * set; };

  if (tid == 0) {
    *s_abort = *reinterpret_cast<volatile unsigned*>(&sync->abort_flag) ? 1 : 0;
#pragma unroll 1
    for (int i = 0; i < L.slots; ++i) { mbar_init(full + 8 * i, 1); mbar_init(empty + 8 * i, kGMma); }
    mbar_init(red_full, kGMma); mbar_init(red_full + 8, kGMma); mbar_init(cleared, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  if (warp >= kGMma) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kGRegsRest));
    if (warp == kGMma + kGAtt) {
      // ------------------------------ weights, in the order the products use them, across steps ------------------------------
      int slot = 0;
      uint32_t par = 0;
      bool ok = true, fresh = true;                            // fresh: first round of the ring, nothing to wait for
      const unsigned char* src = reinterpret_cast<const unsigned char*>(J.packed) + (size_t)cta * L.s.step_bytes;
      // (one copy of the code, rolled: what this warp runs shares the instruction cache with the chain)
#pragma unroll 1
      for (int j = 0; j < n && ok; ++j) {
        const unsigned char* at = src;
#pragma unroll 1
        for (int r = 0; r < nq + 3 && ok; ++r) {               // W_o, W_up, the stretches of W_down, W_k | W_v
          int left = r == 1 ? nt_f : r == nq + 2 ? 2 * nt_d : nt_d;
          const uint32_t tile = r >= 2 && r < nq + 2 ? (uint32_t)(kGMma * 512 * stretch_blocks(L.s, r - 2)) : L.s.tile_d;
#pragma unroll 1
          while (left > 0) {
            if (!fresh) ok = __all_sync(0xffffffffu, ring_wait(empty + 8 * slot, par, sync, s_abort));
            if (!ok) break;
            const uint32_t bar = full + 8 * slot, dst = smem_u32(smem + L.off_ring) + (uint32_t)slot * L.slot_bytes;
            const uint32_t bytes = (uint32_t)(left < kPieceTiles ? left : kPieceTiles) * tile;
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
    // ------------------------------ attention: up to PW (sequence, head) pairs per warp, lanes as dimensions (two each) ------------------------------
    // The pair of position j finishes query j + 1, whose value goes out: that is all the chain waits for.  While the mat-vecs of the next step
    // run, the state of query j + 2 absorbs the pairs of the leaf so far, read back from the caches (every lane reads what it wrote itself;
    // the rows of earlier launches are behind a kernel boundary).
    const int aw = warp - kGMma;
    const bool clears = aw == kGAtt - 1;                       // the warp that sets the CTA's words back (with or without pairs of its own)
    int np = 0;
#pragma unroll
    for (int u = 0; u < PW; ++u) np += cta + (aw + u * kGAtt) * G < pairs ? 1 : 0;
    if (np > 0 || clears) {
      const __nv_bfloat16* q = reinterpret_cast<const __nv_bfloat16*>(J.q);
      __nv_bfloat16 *kc = reinterpret_cast<__nv_bfloat16*>(J.k_cache), *vc = reinterpret_cast<__nv_bfloat16*>(J.v_cache);
      const __nv_bfloat16* g_k = reinterpret_cast<const __nv_bfloat16*>(J.g_k);
      const size_t qrow = (size_t)C.Bs * d;                    // a position's row of q, state and caches
      const bool qkn = (C.norm_flags & RT_NORM_QK) != 0;
      // per pair: its number among the sequences of a row, where its columns, its value and its k|v words lie (a warp with fewer pairs goes through its
      // first one, or any, silently)
      int at_pair[PW], col[PW];
      uint32_t c_at[PW], kv_at[PW];
      float slope[PW], gk0[PW], gk1[PW];
#pragma unroll
      for (int u = 0; u < PW; ++u) {
        const int pair = np == 0 ? cta % pairs : cta + (aw + (u < np ? u : 0) * kGAtt) * G, b = pair / H, h = pair - b * H;
        at_pair[u] = J.b0 * H + pair;
        col[u] = (J.b0 + b) * d + h * kHeadDim + 2 * lane;
        c_at[u] = w_off(b, h * kHeadDim + 2 * lane);
        kv_at[u] = (uint32_t)(b * 2 * d + h * kHeadDim + 2 * lane) * 8u;
        slope[u] = J.alibi ? J.alibi[h] * kLog2e : 0.f;
        gk0[u] = qkn ? gain_at(g_k, h * kHeadDim + 2 * lane) : 1.f;
        gk1[u] = qkn ? gain_at(g_k, h * kHeadDim + 2 * lane + 1) : 1.f;
      }
      float o0[PW], o1[PW], m[PW], l[PW];
      unsigned qw[PW];
      // Iteration j: the pair of position j finishes query j + 1; then query j + 2 absorbs the pairs [key0, t0 + j].  (One copy of the code: it
      // begins two positions early.)
#pragma unroll 1
      for (int j = -2; j < n; ++j) {
        if (j >= 0) {
        const unsigned step = J.steps + (unsigned)j, seq = step + 1u;      // step that reveals position t0 + j
        uint4 ka[PW], va[PW];
        {
          unsigned spins = 0;
          unsigned long long t0 = 0;
          while (true) {
            bool ok = true;
#pragma unroll
            for (int u = 0; u < PW; ++u) {
              const unsigned char* at = w_kv + kv_at[u];
              ka[u] = ld_two_words(at);
              va[u] = ld_two_words(at + (size_t)d * 8);
            }
#pragma unroll
            for (int u = 0; u < PW; ++u) {
              // (a warp without pairs holds nobody up: it may find the pair of a later position, which tells it the same)
              const auto there = [&](unsigned w) { return w == seq || (np == 0 && (int)(w - seq) > 0); };
              ok = ok && there(ka[u].y) && there(ka[u].w) && there(va[u].y) && there(va[u].w);
            }
            if (__all_sync(0xffffffffu, ok)) break;
            if ((++spins & 63u) == 0u && __any_sync(0xffffffffu, group_give_up(sync, s_abort, &t0))) break;
          }
        }
        // Eq. (1): qkRMS over the head, then the storage rounding the cache applies; query j + 1 with this last pair
        unsigned kq[PW], vq[PW];
        float s[PW];
#pragma unroll
        for (int u = 0; u < PW; ++u) {
          const float k0 = __uint_as_float(ka[u].x), k1 = __uint_as_float(ka[u].z);
          const float rk = qkn ? rsqrtf(warp_sum(fmaf(k1, k1, k0 * k0)) * (1.0f / kHeadDim) + C.eps) : 1.0f;
          kq[u] = gpack(k0 * rk * gk0[u], k1 * rk * gk1[u]);
          vq[u] = gpack(__uint_as_float(va[u].x), __uint_as_float(va[u].z));
        }
        if (j + 1 < n) {
#pragma unroll
          for (int u = 0; u < PW; ++u) s[u] = warp_sum(fmaf(ghi(qw[u]), ghi(kq[u]), glo(qw[u]) * glo(kq[u])));
#pragma unroll
          for (int u = 0; u < PW; ++u) {
            const float sc = fmaf(s[u], C.scale_log2, -slope[u]), mn = fmaxf(m[u], sc), corr = exp2f(m[u] - mn), pj = exp2f(sc - mn);
            const float il = 1.0f / fmaf(l[u], corr, pj);
            if (u < np) st_word(c_of(step + 1u) + c_at[u], gpack(fmaf(o0[u], corr, pj * glo(vq[u])) * il, fmaf(o1[u], corr, pj * ghi(vq[u])) * il));
          }
        }
#pragma unroll
        for (int u = 0; u < PW; ++u) {
          if (u < np) {
            const size_t crow = (size_t)(J.t0 + j) * qrow + col[u];
            *reinterpret_cast<unsigned*>(kc + crow) = kq[u];
            *reinterpret_cast<unsigned*>(vc + crow) = vq[u];
            st_word(c_of(step) + c_at[u], kUnset);
          }
        }
        // ---- set back ----
        // k, v of position j come from a CTA that had all of z of this step: every CTA has published its z, so has read all of c, h and g of this step and
        // of z of the one before.  The fence puts c, set back above, before the next but one value of c.  The MMA warps wait for `cleared` and pass a
        // fence before they publish anything of the step after the next; whoever polls these words (in three or four steps) has read such a word and
        // passed a fence of its own in between.
        if (clears) {
          unsigned char *const w_h = c_of(step) + vec, *const w_g = w_h + 2 * (size_t)vec, *const z_before = c_of(step + kTurns - 1u) + 2 * (size_t)vec;
#pragma unroll 1
          for (int b = 0; b < B; ++b) {
            for (int r = lane; r < nd / 2; r += 32) {
              st_word(w_h + w_off(b, d_lo + 2 * r), kUnset);
              st_word(z_before + w_off(b, d_lo + 2 * r), kUnset);
            }
            for (int r = lane; r < nf / 2; r += 32) st_word(w_g + w_off(b, f_lo + 2 * r), kUnset);
          }
        }
        fence_gpu();
        if (clears) {
          __syncwarp();
          if (lane == 0) mbar_arrive(cleared);
        }
        }
        if (j + 2 >= n) continue;
#pragma unroll 1
        for (int u = 0; u < np; ++u) {
          int col_u = col[0], pair_u = at_pair[0];
          float slope_u = slope[0];
#pragma unroll
          for (int w = 1; w < PW; ++w)
            if (w == u) { col_u = col[w]; pair_u = at_pair[w]; slope_u = slope[w]; }
          const int i = j + 2, row = J.t0 - J.row_off + i;
          const size_t at_q = (size_t)row * qrow + col_u, at_s = (size_t)row * C.Bs * H + pair_u;
          const unsigned qv = *reinterpret_cast<const unsigned*>(q + at_q);
          const float2 so = *reinterpret_cast<const float2*>(J.st_o + at_q);
          float a0 = so.x, a1 = so.y, am = J.st_m[at_s], al = J.st_l[at_s];
          const float q0 = glo(qv), q1 = ghi(qv);
          const int key1 = J.t0 + max(j + 1, 0);
#pragma unroll 1
          for (int key = J.key0; key < key1; key += kFoldKeys) {
            unsigned kw[kFoldKeys], vw[kFoldKeys];
#pragma unroll
            for (int e = 0; e < kFoldKeys; ++e) {
              const size_t at = (size_t)min(key + e, key1 - 1) * qrow + col_u;
              kw[e] = __ldcg(reinterpret_cast<const unsigned*>(kc + at));
              vw[e] = __ldcg(reinterpret_cast<const unsigned*>(vc + at));
            }
            float s[kFoldKeys];
#pragma unroll
            for (int e = 0; e < kFoldKeys; ++e) s[e] = fmaf(q1, ghi(kw[e]), q0 * glo(kw[e]));
            // sums over the lanes, transposed: afterwards lanes kFoldLanes e, ... hold the product with key e (the order of sums is warp_sum's)
#pragma unroll
            for (int half = kFoldKeys / 2; half >= 1; half >>= 1) {
              const bool upper = (lane & (kFoldLanes * half)) != 0;
#pragma unroll
              for (int e = 0; e < half; ++e) {
                const float send = upper ? s[e] : s[e + half], keep = upper ? s[e + half] : s[e];
                s[e] = keep + __shfl_xor_sync(0xffffffffu, send, kFoldLanes * half);
              }
            }
#pragma unroll
            for (int off = kFoldLanes / 2; off >= 1; off >>= 1) s[0] += __shfl_xor_sync(0xffffffffu, s[0], off);
            const int mine = key + lane / kFoldLanes, here = min(kFoldKeys, key1 - key);
            const float sc = mine < key1 ? fmaf(s[0], C.scale_log2, -(slope_u * (float)(J.t0 + i - mine))) : -INFINITY;
            // running maximum over the keys, then what each of them multiplies the sums by
            float mx = fmaxf(am, sc);
#pragma unroll
            for (int off = kFoldLanes; off < 32; off <<= 1) {
              const float w = __shfl_up_sync(0xffffffffu, mx, off);
              if (lane >= off) mx = fmaxf(mx, w);
            }
            float before = __shfl_up_sync(0xffffffffu, mx, kFoldLanes);
            if (lane < kFoldLanes) before = am;
            const float corr = exp2f(before - mx), pj = exp2f(sc - mx);
            am = __shfl_sync(0xffffffffu, mx, kFoldLanes * here - 1);
#pragma unroll
            for (int e = 0; e < kFoldKeys; ++e) {
              if (e < here) {
                const float cj = __shfl_sync(0xffffffffu, corr, kFoldLanes * e), pe = __shfl_sync(0xffffffffu, pj, kFoldLanes * e);
                al = fmaf(al, cj, pe);
                a0 = fmaf(a0, cj, pe * glo(vw[e]));
                a1 = fmaf(a1, cj, pe * ghi(vw[e]));
              }
            }
          }
#pragma unroll
          for (int w = 0; w < PW; ++w)
            if (w == u) { o0[w] = a0; o1[w] = a1; m[w] = am; l[w] = al; qw[w] = qv; }
        }
        if (j == -2) {
#pragma unroll
          for (int u = 0; u < PW; ++u) {
            const float il = 1.f / l[u];
            if (u < np) st_word(c_of(J.steps) + c_at[u], gpack(o0[u] * il, o1[u] * il));
          }
        }
      }
    }
    return;
  }

  // ------------------------------ MMA warps (after a wait that ran out they go on to the end) ------------------------------
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kGRegsMma));
  constexpr int kChunk = kGMma / MB;                           // tiles finished together, by one warp per tile and eight sequences
  float2* const red = reinterpret_cast<float2*>(smem + L.off_red);             // [buffer][half of the sequences][tile of the chunk][warp][lane]
  float* const ssq_red = reinterpret_cast<float*>(smem + L.off_ssq);
  const int g = lane >> 2, c = lane & 3;
  const bool pre = (C.norm_flags & RT_NORM_PRE) != 0, kv_norm = pre && !(C.norm_flags & RT_NORM_SKIP_Z);
  const float inv_d = 1.0f / (float)d;
  const int bd = L.s.bd, bf = L.s.bf;
  const int n_bd = max(0, min(bd, (d >> 5) - warp * bd));      // this warp's blocks of d
  const int at_d = n_bd > 0 ? warp * bd : 0;
  const unsigned char* const ring = smem + L.off_ring + g * 64 + c * 16;
  // what this thread finishes: tile u_f of a chunk, sequence b_f, rows 2 c and 2 c + 1 of the tile
  const int u_f = warp % kChunk, half_f = warp / kChunk, b_f = g + 8 * half_f;
  const bool has_f = b_f < B;
  const __nv_bfloat16* const x = reinterpret_cast<const __nv_bfloat16*>(J.x) + (size_t)(has_f ? b_f : 0) * J.x_bs + d_lo;
  __nv_bfloat16* const z = reinterpret_cast<__nv_bfloat16*>(J.z) + (size_t)(has_f ? b_f : 0) * J.z_bs + d_lo;
  int slot = 0;                                                // next ring entry
  uint32_t par = 0;
  unsigned chunk0 = 0;                                         // chunks finished so far (buffers by turns)

#pragma unroll 1
  for (int j = 0; j < n; ++j) {
    const unsigned step = J.steps + (unsigned)j;
    const size_t t = (size_t)(J.t0 + j);
    unsigned char *const w_c = c_of(step), *const w_g = w_c + 3 * (size_t)vec;
    // rows of d: at most four tiles, one chunk.  x_t for the residual, then h, of the rows that this thread finishes
    float2 h = make_float2(0.f, 0.f);
    const int rl_d = u_f * 8 + 2 * c;
    const unsigned xw = has_f && rl_d < nd ? *reinterpret_cast<const unsigned*>(x + t * J.x_ts + rl_d) : 0u;
#pragma unroll 1
    for (int ph = 0; ph < 4; ++ph) {                           // 0: W_o   1: W_up   2: W_down   3: W_k | W_v
      uint4 av[kKP][MB], an[kKP][MB];
      // activations: blocks that this warp and sequences that the job does not have are zeros
      auto start = [&](uint4 (&v)[kKP][MB], int lim) {
#pragma unroll
        for (int i = 0; i < kKP; ++i)
#pragma unroll
          for (int r = 0; r < MB; ++r) {
            const unsigned w = i < lim && g + 8 * r < B ? kUnset : 0u;
            v[i][r] = make_uint4(w, w, w, w);
          }
      };
      auto load = [&](uint4 (&v)[kKP][MB], const unsigned char* base) {      // (all loads on their way before any is looked at)
#pragma unroll
        for (int i = 0; i < kKP; ++i)
#pragma unroll
          for (int r = 0; r < MB; ++r) ld_unset(base + i * 1024 + r * 512, v[i][r]);
      };
      auto g_base = [&](int q) { return w_g + ((size_t)(warp * bf + q * kKP) * 16 + g) * 64 + c * 16; };
      auto g_lim = [&](int q) { return min(stretch_blocks(L.s, q), (dff >> 5) - warp * bf - q * kKP); };
      const unsigned char* base = ph == 2 ? g_base(0) : w_c + (ph == 0 ? 0u : ph == 1 ? vec : 2 * vec) + ((size_t)at_d * 16 + g) * 64 + c * 16;
      start(an, ph == 2 ? g_lim(0) : n_bd);
      load(an, base);

      const int rows = ph == 1 ? nf : nd, tiles = ph == 1 ? nt_f : ph == 3 ? 2 * nt_d : nt_d, n_q = ph == 2 ? nq : 1;
      const bool want_ssq = ph == 1 ? pre : ph == 3 && kv_norm;
      float rs = 1.0f;
      const __nv_bfloat16* const gain = reinterpret_cast<const __nv_bfloat16*>(!want_ssq ? nullptr : ph == 1 ? J.g_mlp : J.g_kv);
      uint2 ga[kKP], gb[kKP];                                  // gains of this thread's columns, fetched before the wait
#pragma unroll
      for (int i = 0; i < kKP; ++i) {
        ga[i] = gb[i] = make_uint2(0u, 0u);
        if (gain && i < n_bd) {
          const __nv_bfloat16* gp = gain + (at_d + i) * 32 + 4 * c;
          ga[i] = *reinterpret_cast<const uint2*>(gp); gb[i] = *reinterpret_cast<const uint2*>(gp + 16);
        }
      }
      // Words of the step before are set back.  Every warp sees that before it contributes to z, without which nobody gets this step's k, v: the clearing warp is
      // never two steps ahead of a waiting warp, whose parity would then mean the wrong one.
      if (ph == 2 && j > 0) ring_wait(cleared, (unsigned)(j - 1) & 1u, sync, s_abort);
      float acc[kQuad][2][4];                                  // W_down: over all stretches
#pragma unroll 1
      for (int q = 0; q < n_q; ++q) {
        const bool last = q + 1 == n_q;
        {
          unsigned spins = 0;
          unsigned long long t0 = 0;
          while (true) {                                       // (the first round of loads is under way)
            unsigned most = 0u;
#pragma unroll
            for (int i = 0; i < kKP; ++i)
#pragma unroll
              for (int r = 0; r < MB; ++r) most = max(most, top(an[i][r]));
            if (__all_sync(0xffffffffu, most != kUnset)) break;
            if ((++spins & 63u) == 0u && __any_sync(0xffffffffu, group_give_up(sync, s_abort, &t0))) break;
            load(an, base);
          }
#pragma unroll
          for (int i = 0; i < kKP; ++i)
#pragma unroll
            for (int r = 0; r < MB; ++r) av[i][r] = an[i][r];
        }
        if (!last) { base = g_base(q + 1); start(an, g_lim(q + 1)); load(an, base); }
        if (want_ssq) {
#pragma unroll
          for (int r = 0; r < MB; ++r) {
            float sq = 0.f;
#pragma unroll
            for (int i = 0; i < kKP; ++i) {
              uint4& v = av[i][r];
              const float e0 = glo(v.x), e1 = ghi(v.x), e2 = glo(v.y), e3 = ghi(v.y), e4 = glo(v.z), e5 = ghi(v.z), e6 = glo(v.w), e7 = ghi(v.w);
              sq += fmaf(e3, e3, fmaf(e2, e2, fmaf(e1, e1, e0 * e0)));
              sq += fmaf(e7, e7, fmaf(e6, e6, fmaf(e5, e5, e4 * e4)));
              if (gain) {
                v.x = gpack(e0 * glo(ga[i].x), e1 * ghi(ga[i].x)); v.y = gpack(e2 * glo(ga[i].y), e3 * ghi(ga[i].y));
                v.z = gpack(e4 * glo(gb[i].x), e5 * ghi(gb[i].x)); v.w = gpack(e6 * glo(gb[i].y), e7 * ghi(gb[i].y));
              }
            }
            sq += __shfl_xor_sync(0xffffffffu, sq, 1); sq += __shfl_xor_sync(0xffffffffu, sq, 2);
            if (c == 0) ssq_red[warp * 16 + 8 * r + g] = sq;
          }
        }
        // where this warp's blocks lie in a tile of this stretch (blocks beyond it read the last one: they multiply zeros)
        const int nb = ph == 2 ? stretch_blocks(L.s, q) : bd, lim = ph == 2 ? nb : max(1, n_bd);
        const uint32_t tile = ph == 2 ? (uint32_t)(kGMma * 512 * nb) : L.s.tile_d;
        const unsigned char* const ring_q = ring + (ph == 2 ? warp * nb : at_d) * 512;
        uint32_t off[kKP];
#pragma unroll
        for (int i = 0; i < kKP; ++i) off[i] = (uint32_t)(i < lim ? i : lim - 1) * 512u;
        // ---- products, four tiles at a time; while they run, this warp's part of the chunk before is finished ----
        int pending = -1;
#pragma unroll 1
        for (int ti = 0;; ti += kQuad) {
          const bool more = ti < tiles;
          if (more) {
            const int slot2 = slot + 1 == L.slots ? 0 : slot + 1;
            const bool two = ti + kPieceTiles < tiles;
            ring_wait(full + 8 * slot, par, sync, s_abort);
            if (two) ring_wait(full + 8 * slot2, slot2 ? par : par ^ 1, sync, s_abort);
            const unsigned char* const w0 = ring_q + (uint32_t)slot * L.slot_bytes;
            const unsigned char* const w1 = two ? ring_q + (uint32_t)slot2 * L.slot_bytes : w0;      // (products of tiles that do not exist are not used)
            if (q == 0) {
#pragma unroll
              for (int u = 0; u < kQuad; ++u)
#pragma unroll
                for (int e = 0; e < 4; ++e) { acc[u][0][e] = 0.f; acc[u][1][e] = 0.f; }
            }
#pragma unroll
            for (int i = 0; i < kKP; ++i) {                    // (no branch around a product: blocks beyond the stretch multiply zeros)
              uint4 w[kQuad];
#pragma unroll
              for (int u = 0; u < kQuad; ++u) w[u] = *reinterpret_cast<const uint4*>((u < kPieceTiles ? w0 : w1) + ((u & 1) ? tile : 0u) + off[i]);
#pragma unroll
              for (int u = 0; u < kQuad; ++u)
                gmma(acc[u][0], av[i][0].x, MB == 2 ? av[i][MB - 1].x : 0u, av[i][0].y, MB == 2 ? av[i][MB - 1].y : 0u, w[u].x, w[u].y);
#pragma unroll
              for (int u = 0; u < kQuad; ++u)
                gmma(acc[u][1], av[i][0].z, MB == 2 ? av[i][MB - 1].z : 0u, av[i][0].w, MB == 2 ? av[i][MB - 1].w : 0u, w[u].z, w[u].w);
            }
            __syncwarp();
            if (lane == 0) { mbar_arrive(empty + 8 * slot); if (two) mbar_arrive(empty + 8 * slot2); }
            slot = two ? slot2 : slot;
            if (two && slot2 == 0) par ^= 1;
            if (++slot == L.slots) { slot = 0; par ^= 1; }
          }
          if (pending >= 0) {
            // sums over the eight warps, one (tile, eight sequences) per warp
            const unsigned at = chunk0 + (unsigned)pending;
            ring_wait(red_full + 8 * (at & 1u), (at >> 1) & 1u, sync, s_abort);
            const float2* src = red + (at & 1u) * (kGMma * kGMma * 32) + ((half_f * kChunk + u_f) * kGMma) * 32 + lane;
            float2 v[kGMma];
#pragma unroll
            for (int w = 0; w < kGMma; ++w) v[w] = src[w * 32];
            if (want_ssq && pending == 0) {
              float s = 0.f;
#pragma unroll
              for (int w = 0; w < kGMma; ++w) s += ssq_red[w * 16 + b_f];
              rs = rsqrtf(s * inv_d + C.eps);
            }
            float y0 = 0.f, y1 = 0.f;
#pragma unroll
            for (int w = 0; w < kGMma; ++w) { y0 += v[w].x; y1 += v[w].y; }
            const int tf = pending * kChunk + u_f;
            const bool second = ph == 3 && tf >= nt_d;
            const int rl = (second ? tf - nt_d : tf) * 8 + 2 * c;
            if (tf < tiles && rl < rows && has_f) {
              if (ph == 3) {                                   // raw k_t, v_t from RMS(z_t): Eqs. (1)-(2) before qkRMS
                st_flag2(w_kv + (uint32_t)(b_f * 2 * d + (second ? d : 0) + d_lo + rl) * 8u, __float_as_uint(y0 * rs), __float_as_uint(y1 * rs), step + 1u);
              } else {
                unsigned word;
                if (ph == 1) {                                 // g = GELU(W_up RMS(h))
                  auto gelu = [](float v) { return 0.5f * v * (1.0f + erff(v * 0.70710678118654752f)); };
                  word = gpack(gelu(y0 * rs), gelu(y1 * rs));
                } else {                                       // h = x_t + alpha W_o c_t, then z_t = h + alpha W_down g   (layer output)
                  h = make_float2((ph == 0 ? glo(xw) : h.x) + C.alpha * y0, (ph == 0 ? ghi(xw) : h.y) + C.alpha * y1);
                  word = gpack(h.x, h.y);
                  if (ph == 2) *reinterpret_cast<unsigned*>(z + t * J.z_ts + rl) = word;
                }
                st_word(w_c + (ph == 0 ? vec : ph == 1 ? 3 * vec : 2 * vec) + w_off(b_f, (ph == 1 ? f_lo : d_lo) + rl), word);
              }
            }
            pending = -1;
          }
          if (!more || !last) break;                           // (W_down: its only tiles go on with the next stretch)
          // (four tiles are of one chunk; what tiles that do not exist leave there is not used)
          float2* const dst = red + ((chunk0 + (unsigned)(ti / kChunk)) & 1u) * (kGMma * kGMma * 32) + ((ti % kChunk) * kGMma + warp) * 32 + lane;
#pragma unroll
          for (int u = 0; u < kQuad; ++u) {
#pragma unroll
            for (int r = 0; r < MB; ++r) {
              const float2 v = make_float2(acc[u][0][2 * r] + acc[u][1][2 * r], acc[u][0][2 * r + 1] + acc[u][1][2 * r + 1]);
              dst[(u + r * kChunk) * (kGMma * 32)] = v;
            }
          }
          if ((ti + kQuad) % kChunk == 0 || ti + kQuad >= tiles) {
            __syncwarp();
            pending = ti / kChunk;
            if (lane == 0) mbar_arrive(red_full + 8 * ((chunk0 + (unsigned)pending) & 1u));
          }
        }
      }
      chunk0 += (unsigned)((tiles + kChunk - 1) / kChunk);
    }
    fence_gpu();
  }
}

}  // namespace

// SMs of a group; every CTA owns rows of W_down (what the words are set back by: whoever publishes z has read all that came before).
static int group_size(int d, int places) { const int g = kB200Sms / places; return g < d / 2 ? g : d / 2; }

// Microseconds per position, estimated: the exchanges, and the rounds of four tiles that a warp goes through.  Measured / estimated for 2, 4, 6, 8 places (d = 768 six, d = 1024
// four at most, see leaf_group_shape): B = 1 d = 512 11.9 / 12.4, 12.0 / 12.6, 13.5 / 13.1, 14.3 / 13.3; d = 768 14.1 / 13.6, 15.0 / 14.4, 14.8 / 14.7; d = 1024 14.5 / 14.9, 16.5 / 16.4;
// B = 16 d = 512 14.4 / 14.4, 14.1 / 14.8, 15.3 / 15.5, 16.6 / 15.9; d = 768 16.7 / 16.5, 17.4 / 17.6, 18.1 / 18.2; d = 1024 17.8 / 18.6, 19.8 / 20.8.
float leaf_group_step_us(int B, int d, int dff, int places) {
  const GroupShape s = group_shape(d, dff, group_size(d, places));
  auto rounds = [](int tiles) { return (tiles + kQuad - 1) / kQuad; };
  const float n = (float)((1 + s.nq + rounds(s.nt_f) + rounds(2 * s.nt_d)) * d), b = 0.2f * (float)B;
  return B > 8 ? 9.3f + b + 7.4e-4f * n : 11.0f + b + 4.6e-4f * n;
}

size_t leaf_group_words_bytes(int d, int dff) { return align_up((size_t)kTurns * (3 * 32 * d + 32 * dff) + (size_t)16 * 2 * d * 8, 256); }
size_t leaf_group_packed_bytes(int d, int dff, int places) {
  const int g = group_size(d, places);
  return align_up((size_t)g * group_shape(d, dff, g).step_bytes, 256);
}

// Whether jobs of B sequences run on groups of 148 / places SMs (pure arithmetic).  A CTA's rows of d are at most kQuad tiles, so that one pass finishes them: d = 1024
// takes four places at most, 768 six, 576 and less eight.
bool leaf_group_shape(int B, int d, int H, int dff, int places, size_t max_smem) {
  if (B < 1 || B > 16 || places < 1 || places > kGroupJobs || d % 64 || d > 1024 || dff % 32 || dff > 8 * d) return false;
  const int g = group_size(d, places);
  if (B * H > kMaxPairs * kGAtt * g || group_shape(d, dff, g).nt_d > kQuad) return false;
  return group_layout(d, dff, g, max_smem).slots >= 4;
}

cudaError_t leaf_group_pack(const GroupPackLayer* layers, int n, int d, int dff, int places, cudaStream_t s) {
  const int g = group_size(d, places);
  for (int l0 = 0; l0 < n; l0 += kGroupPackLayers) {
    GroupPackArgs a;
    memset(&a, 0, sizeof(a));
    a.d = d; a.dff = dff; a.g = g;
    const int here = n - l0 < kGroupPackLayers ? n - l0 : kGroupPackLayers;
    for (int i = 0; i < here; ++i) a.layer[i] = layers[l0 + i];
    const GroupShape sh = group_shape(d, dff, g);
    group_pack_kernel<<<dim3(g, 3 * sh.nt_d + sh.nt_f + sh.nt_d * sh.nq, here), 256, 0, s>>>(a);
  }
  return cudaGetLastError();
}

cudaError_t leaf_group_launch(const GroupCommon& c, const GroupJob* jobs, int n_jobs, int places, cudaStream_t s) {
  GroupArgs a;
  memset(&a, 0, sizeof(a));
  a.c = c; a.n_jobs = n_jobs; a.gsize = group_size(c.d, places);
  int most = 0;
  for (int i = 0; i < n_jobs; ++i) { a.job[i] = jobs[i]; most = jobs[i].B > most ? jobs[i].B : most; }
  GroupLayout L = group_layout(c.d, c.dff, a.gsize, kB200SmemPerCta);
  const int pw = ceil_div(ceil_div(most * c.H, a.gsize), kGAtt);
  auto pick = [&](auto mb) -> const void* {
    constexpr int MB = decltype(mb)::value;
    return pw <= 1 ? (const void*)&leaf_group_kernel<MB, 1> : pw == 2 ? (const void*)&leaf_group_kernel<MB, 2> : (const void*)&leaf_group_kernel<MB, 3>;
  };
  const void* fn = most > 8 ? pick(std::integral_constant<int, 2>{}) : pick(std::integral_constant<int, 1>{});
  cudaError_t e = ensure_dynamic_smem(fn, (int)L.total);
  if (e != cudaSuccess) return e;
  void* args[] = {(void*)&a, (void*)&L};
  return cudaLaunchCooperativeKernel(fn, dim3(a.gsize * n_jobs), dim3(kGThreads), args, L.total, s);
}

}  // namespace rt
