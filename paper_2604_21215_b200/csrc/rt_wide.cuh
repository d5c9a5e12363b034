// Parts of the persistent loops of wide batches (rt_wide_loop.cu, rt_wide_backward.cu): a group of SMs runs a chain of tcgen05 products and
// row-wise steps over at most 128 sequences.  Warp 0 fetches operands and watches the group's counters, warp 1 issues the products, eight warps
// do the row work.
#pragma once
#include "rt_gelu.h"
#include "rt_kernels.h"
#include "rt_tc.cuh"

namespace rt {

constexpr int kWThreads = 320, kWEpi = 256;
constexpr int kWBlocks = 2;                                // 64-wide blocks of A and of W per fill of the operand ring
constexpr uint32_t kWRing = 192512;
constexpr int kWSlotsMax = 11;
constexpr int kWStagePitch = 36;                           // floats per row of a warp's 32 x 32 staging area
constexpr uint32_t kWStage = kWRing, kWStageWarp = 32 * kWStagePitch * 4;
constexpr uint32_t kWBars = kWStage + 8 * kWStageWarp, kWTmem = kWBars + 256, kWAbort = kWTmem + 8, kWTotal = kWAbort + 8;
constexpr int kWBuf = 128;                                 // TMEM columns per accumulator, two of them
constexpr int kWCounterStride = 32;                        // unsigned words between counters
constexpr int kWMaxSteps = 8;

// (for global memory only: over all state spaces the fence took 0.5 us longer, a tenth of a step)
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ bool epi_all(bool ok) {         // barrier of the eight row warps; true when all of them are fine
  int r;
  asm volatile("{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n barrier.cta.red.and.pred q, 1, 256, p;\n selp.b32 %0, 1, 0, q;\n}" : "=r"(r) : "r"((int)ok) : "memory");
  return r != 0;
}
__device__ __forceinline__ void unpack8(const uint4& w, float (&f)[8]) {
  const unsigned a[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) { f[2 * i] = __uint_as_float(a[i] << 16); f[2 * i + 1] = __uint_as_float(a[i] & 0xffff0000u); }
}
__device__ __forceinline__ unsigned pack2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const unsigned*>(&v);
}
__device__ __forceinline__ uint4 ldcg16(const __nv_bfloat16* p) { return __ldcg(reinterpret_cast<const uint4*>(p)); }
__device__ __forceinline__ float sum8(float v) {           // over the eight lanes of a (sequence, head)
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  return v;
}
__device__ __forceinline__ float erfc_step(float x) {      // t of rt_gelu.h
  float t;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t) : "f"(fmaf(kErfcSlope, fabsf(x), 1.0f)));
  return t;
}
__device__ __forceinline__ float gelu_wide(float x) { return gelu_of(x, erfc_step(x), ex2(x * x * (-0.5f * kLog2e))); }

static __device__ __noinline__ bool wide_wait(uint32_t bar, uint32_t parity, volatile int* s_abort, SyncArea* sync) { return warp_mbar_wait(bar, parity, s_abort, sync); }

// Where a CTA stands and how its group meets.
struct WideCta {
  unsigned char* smem;
  uint32_t sbase;
  volatile int* s_abort;
  SyncArea* sync;
  unsigned* counters;                                      // of this group
  int rank, G, arank;                                      // arank: rank in the attention step, which begins with the CTAs that have no tile of the step before
  __device__ uint32_t full(int s) const { return sbase + kWBars + 8u * (uint32_t)s; }
  __device__ uint32_t empty(int s) const { return sbase + kWBars + 8u * (uint32_t)(kWSlotsMax + s); }
  __device__ uint32_t tfull(int b) const { return sbase + kWBars + 8u * (uint32_t)(2 * kWSlotsMax + b); }
  __device__ uint32_t tempty(int b) const { return sbase + kWBars + 8u * (uint32_t)(2 * kWSlotsMax + 2 + b); }
  __device__ uint32_t flag() const { return sbase + kWBars + 8u * (uint32_t)(2 * kWSlotsMax + 4); }
  // warp 0: until `target` CTAs have counted themselves in at a step
  __device__ bool poll(int step, unsigned target) const {
    const unsigned* c = counters + step * kWCounterStride;
    unsigned spins = 0;
    unsigned long long t_start = 0;
    bool ok = true;
    while (ld_acquire_u32(c) < target) {
      if ((++spins & 1023u) == 0u) {
        if (*s_abort || *reinterpret_cast<volatile unsigned*>(&sync->abort_flag)) { ok = false; break; }
        const unsigned long long now = globaltimer_ns();
        if (t_start == 0) t_start = now;
        else if (now - t_start > kWaitLimitNs) {
          sync->status = RT_ERR_TIMEOUT;
          __threadfence();
          atomicExch(&sync->abort_flag, 1u);
          ok = false;
          break;
        }
      }
    }
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) *s_abort = 1;
    fence_async_proxy();
    return ok;
  }
};

// Operand fetches of one product step: the weights of the first blocks, then (after the wait) their operand rows, then the rest block by block.
// emask / fmask: parity of the next wait on a slot's empty barrier / of the latest fill of a slot.
// A copy of up to 16 KB costs an SM about 90 ns whatever its size, so a copy covers two blocks (a three-dimensional map: 64 columns, rows,
// blocks): a 128-column tile over 1024 takes 4.8 us that way and 5.8 us with single blocks, although more of those are under way.
struct WideFetch { uint32_t emask, fmask; };
template <typename Wait>
__device__ __forceinline__ bool wide_fetch(const WideCta& c, WideFetch& f, const WideStage& st, const CUtensorMap* ma, const CUtensorMap* mw, const CUtensorMap* mw2, int m0,
                                           uint32_t a_bytes, Wait wait) {
  const uint32_t w_bytes = (uint32_t)st.bn * 128u, slot_bytes = kWBlocks * (a_bytes + w_bytes);
  bool ok = true, waited = false;
#pragma unroll 1
  for (int job = c.rank; job < st.tiles * st.splits && ok; job += c.G) {
    const int tile = job % st.tiles, split = job / st.tiles;
    const int k0 = st.fills * split / st.splits, n = st.fills * (split + 1) / st.splits - k0;
    const bool second = mw2 && tile >= st.tiles / 2;
    const CUtensorMap* w = second ? mw2 : mw;
    const int n0 = (second ? tile - st.tiles / 2 : tile) * st.bn;
    const int pre = n < st.slots ? n : st.slots;
#pragma unroll 1
    for (int k = 0; k < pre; ++k) {
      expect_tx_elect(c.full(k), slot_bytes);
      tma_load_3d(c.sbase + k * slot_bytes + kWBlocks * a_bytes, w, c.full(k), 0, n0, kWBlocks * (k0 + k));
      f.fmask ^= 1u << k;
    }
    if (!waited) { ok = wait(); waited = true; }
#pragma unroll 1
    for (int k = 0; k < pre; ++k) tma_load_3d(c.sbase + k * slot_bytes, ma, c.full(k), 0, m0, kWBlocks * (k0 + k));      // (given up or not: the fill has to land)
    int s = 0;
#pragma unroll 1
    for (int k = pre; k < n && ok; ++k) {
      ok = wide_wait(c.empty(s), (f.emask >> s) & 1u, c.s_abort, c.sync);
      if (!ok) break;
      f.emask ^= 1u << s;
      f.fmask ^= 1u << s;
      expect_tx_elect(c.full(s), slot_bytes);
      tma_load_3d(c.sbase + s * slot_bytes, ma, c.full(s), 0, m0, kWBlocks * (k0 + k));
      tma_load_3d(c.sbase + s * slot_bytes + kWBlocks * a_bytes, w, c.full(s), 0, n0, kWBlocks * (k0 + k));
      if (++s == st.slots) s = 0;
    }
#pragma unroll 1
    for (int j = 0; j < pre && ok; ++j) {                  // every slot read: the next product lays the ring out anew
      ok = wide_wait(c.empty(j), (f.emask >> j) & 1u, c.s_abort, c.sync);
      if (ok) f.emask ^= 1u << j;
    }
    if (!ok) {
      // gave up: the fills under way have to land before the shared memory goes away (bounded).  fmask holds the parity AFTER the fill.
#pragma unroll 1
      for (int j = 0; j < pre; ++j) {
        unsigned spins = 0;
        while (!mbar_try_wait(c.full(j), ((f.fmask >> j) & 1u) ^ 1u) && ++spins < (1u << 20)) {}
      }
    }
  }
  return ok;
}

// The products of one step.
struct WideIssue { uint32_t fmask; int jobs; };
__device__ __forceinline__ bool wide_issue(const WideCta& c, WideIssue& w, const WideStage& st, uint32_t a_bytes, uint32_t tmem) {
  const uint32_t w_bytes = (uint32_t)st.bn * 128u, slot_bytes = kWBlocks * (a_bytes + w_bytes), idesc = make_idesc(st.bn, false);
  bool ok = true;
#pragma unroll 1
  for (int job = c.rank; job < st.tiles * st.splits && ok; job += c.G) {
    const int split = job / st.tiles;
    const int n = st.fills * (split + 1) / st.splits - st.fills * split / st.splits;
    const int buf = w.jobs & 1;
    if (w.jobs >= 2) ok = wide_wait(c.tempty(buf), ((w.jobs >> 1) - 1) & 1, c.s_abort, c.sync);
    int s = 0;
#pragma unroll 1
    for (int k = 0; k < n && ok; ++k) {
      ok = wide_wait(c.full(s), (w.fmask >> s) & 1u, c.s_abort, c.sync);
      if (!ok) break;
      w.fmask ^= 1u << s;
      tc_fence_after();
#pragma unroll
      for (int j = 0; j < kWBlocks; ++j) {
        const uint64_t a0 = make_desc(c.sbase + s * slot_bytes + j * a_bytes, 16, 1024), b0 = make_desc(c.sbase + s * slot_bytes + kWBlocks * a_bytes + j * w_bytes, 16, 1024);
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) tc_mma(tmem + (uint32_t)(buf * kWBuf), a0 + 2u * ks, b0 + 2u * ks, idesc, (k > 0 || j > 0 || ks > 0) ? 1u : 0u);
      }
      tc_commit(c.empty(s));
      if (++s == st.slots) s = 0;
    }
    if (ok) tc_commit(c.tfull(buf));
    ++w.jobs;
  }
  return ok;
}

// An accumulator block of 32 rows and 32 columns through the warp's staging area: rows belong to lanes in TMEM, and storing them that way
// touches 32 lines per instruction (the stores of a 128 x 128 fp32 tile took 2.6 us); afterwards eight lanes hold a row, four columns each.
// f is applied to every entry on the way (by the lane of its row, 32 independent entries).
template <typename F>
__device__ __forceinline__ void wide_stage(float* st, uint32_t taddr, int lane, F f) {
  uint32_t r[32];
  tc_ld32(taddr, r);
  tc_wait_ld();
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 8; ++i)
    *reinterpret_cast<float4*>(st + lane * kWStagePitch + 4 * i) =
        make_float4(f(__uint_as_float(r[4 * i])), f(__uint_as_float(r[4 * i + 1])), f(__uint_as_float(r[4 * i + 2])), f(__uint_as_float(r[4 * i + 3])));
  __syncwarp();
}

__device__ __forceinline__ int wide_active_rows(int units, int per_cta, int G) {
  const int n = (units + per_cta - 1) / per_cta;
  return n < G ? n : G;
}
__device__ __forceinline__ int wide_active(const WideStage& st, int G) { return st.tiles * st.splits < G ? st.tiles * st.splits : G; }

// Barriers and accumulators of a CTA; the whole CTA calls both.
__device__ __forceinline__ void wide_setup(const WideCta& c, int tid, int warp) {
  if (tid == 0) {
    *c.s_abort = 0;
    for (int s = 0; s < kWSlotsMax; ++s) { mbar_init(c.full(s), 1); mbar_init(c.empty(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(c.tfull(b), 1); mbar_init(c.tempty(b), 8); }
    mbar_init(c.flag(), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(c.sbase + kWTmem), "n"(2 * kWBuf) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
}
__device__ __forceinline__ void wide_teardown(uint32_t tmem, int warp) {
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(2 * kWBuf) : "memory");
  }
}

// ---- host ----
inline WideStage wide_stage_of(int n, int k, int bn, int splits, int a_bytes) {
  WideStage st;
  st.bn = bn; st.tiles = n / bn; st.splits = splits;
  st.fills = k / 64 / kWBlocks;
  st.slots = (int)(kWRing / (kWBlocks * ((unsigned)a_bytes + (unsigned)bn * 128u)));
  if (st.slots > kWSlotsMax) st.slots = kWSlotsMax;
  return st;
}
// A product of n columns over k on G CTAs, not split: the narrowest tile that gives every CTA at most one (d and d_ff are multiples of 128).
inline WideStage stage_whole(int n, int k, int G, int a_bytes, int bn_max) { return wide_stage_of(n, k, bn_max == 128 && n / 64 > G ? 128 : 64, 1, a_bytes); }
// The same in parts of the contraction, summed by a row step: the operand rows of a part, not its weights, are what a CTA waits for, so as
// many parts (of at least four blocks, at most eight) as the group has CTAs for; tiles of 64 columns where the group is large enough.
inline WideStage stage_split(int n, int k, int G, int a_bytes) {
  const int bn = (n / 64) * 8 <= G ? 64 : 128;
  int sp = G / (n / bn);
  if (sp > 8) sp = 8;
  if (sp > k / 256) sp = k / 256;
  return wide_stage_of(n, k, bn, sp < 1 ? 1 : sp, a_bytes);
}
// [rows, cols] bf16 as blocks of 64 columns: a box is two blocks of box_rows rows
inline bool map_blocks(CUtensorMap* out, const void* base, long long rows, int cols, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[3] = {64, (cuuint64_t)rows, (cuuint64_t)(cols / 64)}, strides[2] = {(cuuint64_t)cols * 2, 128};
  const cuuint32_t box[3] = {64u, (cuuint32_t)box_rows, (cuuint32_t)kWBlocks}, estr[3] = {1, 1, 1};
  return fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace rt
