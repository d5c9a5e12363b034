// Reverse loop of wide batches (up to 128 sequences per group of SMs), one cooperative launch per leaf, bf16: the counterpart of
// rt_wide_loop.cu, same roles, barriers and operand ring.  A position is seven steps (the launches of rt_backward.cu's wide_position_tc):
//   P1 [dk_raw | dv] [W_k; W_v] in parts    R1 dr = sum, Gz = dz + RMS backward through z
//   P2 (alpha Gz) W_down, times GELU'       P3 dpre W_up in parts    R3 du = sum, dh = Gz + RMS backward through h
//   P4 dc = (alpha dh) W_o                  A  the pairs of the leaf, the temporary pair, the operand of the position before
// R1 and R3 need sums over whole rows: four warps own a row.  In A only the newest pair, i - 1, is on the chain; the leaf's older pairs are
// updated after the step has been counted in, by the same threads at every position.
//
// Measured per position at d = 1024, d_ff = 4096: B = 96 36 us (63 as seven launches, 74 as fifteen), B = 512 75 (106); three-term operands B = 16 32
// (43 in two slices of the mat-vec kernel), B = 32 33 (84 in four).  A step is about 5 us, as in the forward loop.
#include <type_traits>

#include "rt_bwd.cuh"
#include "rt_wide.cuh"

namespace rt {
namespace {

enum { B_KV = 0, B_RZ = 1, B_DOWN = 2, B_UP = 3, B_RH = 4, B_OUT = 5, B_ATTN = 6, B_STEPS = 7 };
// The products in order (indices of WideBwdParams::st): W_k | W_v, W_down, W_up, W_o (all transposed).
struct WideBwdMaps { CUtensorMap a[4], w[4]; };

__device__ __forceinline__ float gelu_grad_wide(float x) { return gelu_grad_of(x, erfc_step(x), ex2(x * x * (-0.5f * kLog2e))); }
__device__ __forceinline__ F8 ldcg8(const float* p) {
  const float4 a = __ldcg(reinterpret_cast<const float4*>(p)), b = __ldcg(reinterpret_cast<const float4*>(p + 4));
  return F8{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}

// CH: groups of four columns per thread of a row's four warps (d <= 512 CH).  TERMS = 3: at most 32 sequences whose operands are three bf16
// terms each (2^-24 of the value): rows 0 .. 31, 32 .. 63 and 64 .. 95 of the row tile, so a product costs what it does anyway, and the row
// warps add the three accumulator quadrants through their staging areas.
template <int CH, int TERMS>
__global__ void __launch_bounds__(kWThreads, 1) wide_backward_kernel(const __grid_constant__ WideBwdMaps maps, const __grid_constant__ WideBwdParams p, const __grid_constant__ AttnBufs a,
                                                                     const __grid_constant__ WidePair wp) {
  extern __shared__ unsigned char smem_raw[];
  WideCta c;
  c.smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  c.sbase = smem_u32(c.smem);
  c.s_abort = reinterpret_cast<volatile int*>(c.smem + kWAbort);
  c.sync = p.sync;
  c.G = p.G;
  const int group = blockIdx.x / p.G;
  c.rank = blockIdx.x % p.G;
  c.arank = c.rank;
  c.counters = p.counters + group * kWMaxSteps * kWCounterStride;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int m0 = group * p.R, R = p.B - m0 < p.R ? p.B - m0 : p.R;
  wide_setup(c, tid, warp);
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(c.smem + kWTmem), a_bytes = (uint32_t)p.a_bytes;
  const int d = p.d, H = p.H, units = R * H;
  auto active_of = [&](int step) {
    if (step == B_RZ || step == B_RH) return R < p.G ? R : p.G;
    if (step == B_ATTN) return wide_active_rows(units, 4, p.G);
    return wide_active(p.st[step == B_KV ? 0 : step == B_OUT ? 3 : step - 1], p.G);
  };
  if (warp == 0) {
    WideFetch f = {0u, 0u};
    bool ok = true;
#pragma unroll 1
    for (int i = p.e0 - 1; i >= p.s0 && ok; --i) {
      const unsigned n = p.steps + (unsigned)(p.e0 - 1 - i);                 // positions done before this one
      int product = 0;
#pragma unroll 1
      for (int step = 0; step < B_STEPS && ok; ++step) {
        const bool rows = step == B_RZ || step == B_RH || step == B_ATTN;
        auto wait = [&]() {
          bool r = true;
          if (step == B_KV) { if (i < p.e0 - 1) r = c.poll(B_ATTN, n * (unsigned)active_of(B_ATTN)); }
          else r = c.poll(step - 1, (n + 1) * (unsigned)active_of(step - 1));
          if (lane == 0 && r) mbar_arrive(c.flag());
          __syncwarp();
          return r;
        };
        if (c.rank < active_of(step)) {
          if (rows) ok = wait();
          else ok = wide_fetch(c, f, p.st[product], &maps.a[product], &maps.w[product], nullptr, m0, a_bytes, wait);
        }
        if (!rows) ++product;
      }
    }
  } else if (warp == 1) {
    WideIssue w = {0u, 0};
    bool ok = true;
#pragma unroll 1
    for (int i = p.e0 - 1; i >= p.s0 && ok; --i)
#pragma unroll 1
      for (int product = 0; product < 4 && ok; ++product) ok = wide_issue(c, w, p.st[product], a_bytes, tmem);
  } else {
    const int ew = warp - 2, quad = warp & 3, half = ew >> 2;
    const uint32_t t_row = tmem + ((uint32_t)(quad * 32) << 16);
    const size_t rstride = (size_t)p.B * d;
    float* stage = reinterpret_cast<float*>(c.smem + kWStage + ew * kWStageWarp);
    uint32_t flags = 0;
    int jobs = 0;
    auto flag_wait = [&]() { const bool r = wide_wait(c.flag(), flags & 1u, c.s_abort, c.sync); ++flags; return r; };
    auto acc_wait = [&]() {
      const bool r = wide_wait(c.tfull(jobs & 1), (jobs >> 1) & 1, c.s_abort, c.sync);
      tc_fence_after();
      return r;
    };
    auto acc_done = [&]() {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(c.tempty(jobs & 1));
      ++jobs;
    };
    auto finish = [&](bool ok, int step) {
      ok = epi_all(ok);
      if (tid == 64 && ok) red_release_add_u32(c.counters + step * kWCounterStride, 1u);
      return ok;
    };
    constexpr int kIter = TERMS == 3 ? 2 : 8;              // rows of a staged block per warp: all 32 of its own quadrant, or 8 of the 32 sequences
    const int row_base = TERMS == 3 ? 8 * (ew & 3) : 0, row_of0 = TERMS == 3 ? 0 : quad * 32;
    auto team_all = [&](bool ok) {                             // the four warps of a half agree (and have staged their blocks)
      int r;
      asm volatile("{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n barrier.cta.red.and.pred q, %2, 128, p;\n selp.b32 %0, 1, 0, q;\n}" : "=r"(r) : "r"((int)ok), "r"(2 + half) : "memory");
      return r != 0;
    };
    // columns [cc, cc + 32) of the accumulator: f(sequence of the group, column of the block, values), called by every lane kIter times; false when
    // the accumulator never came
    auto staged = [&](bool good, int cc, auto f) {
      if (good) wide_stage(stage, t_row + (uint32_t)((jobs & 1) * kWBuf + cc), lane, [](float v) { return v; });
      if (TERMS == 3) good = team_all(good);
      if (!good) return false;
      const float* base = reinterpret_cast<const float*>(c.smem + kWStage);
#pragma unroll
      for (int k = 0; k < kIter; ++k) {
        const int r = row_base + 4 * k + (lane >> 3), at = r * kWStagePitch + 4 * (lane & 7);
        float4 v;
        if (TERMS == 3) {                                      // quadrant q belongs to warp (q + 2) & 3 of the half
          const float4 x = *reinterpret_cast<const float4*>(base + (2 + 4 * half) * (kWStageWarp / 4) + at), y = *reinterpret_cast<const float4*>(base + (3 + 4 * half) * (kWStageWarp / 4) + at),
                       z = *reinterpret_cast<const float4*>(base + (0 + 4 * half) * (kWStageWarp / 4) + at);
          v = make_float4(x.x + (y.x + z.x), x.y + (y.y + z.y), x.z + (y.z + z.z), x.w + (y.w + z.w));
        } else {
          v = *reinterpret_cast<const float4*>(stage + at);
        }
        f(k, row_of0 + r, 4 * (lane & 7), v);
      }
      if (TERMS == 3) team_all(true);                          // (read before the next block is staged)
      return true;
    };
    // a product whose sums (or parts of them) go to memory as they are: out[split][row][column]
    auto plain_product = [&](const WideStage& st, float* out) {
      bool good = flag_wait();
#pragma unroll 1
      for (int job = c.rank; job < st.tiles * st.splits; job += c.G) {
        const int n0 = (job % st.tiles) * st.bn, split = job / st.tiles;
        if (good) good = acc_wait();
#pragma unroll 1
        for (int cc = half * (st.bn >> 1); cc < (half + 1) * (st.bn >> 1); cc += 32) {
          const bool done = staged(good, cc, [&](int, int rr, int col, const float4& v) {
            if (rr < R) *reinterpret_cast<float4*>(out + ((size_t)split * p.B + m0 + rr) * d + n0 + cc + col) = v;
          });
          good = good && done;
        }
        if (!good) break;
        acc_done();
      }
      return good;
    };
    // out = add + RMS backward of the sum of the parts through RMS(u) g; keeps the sum, leaves bf16(alpha out) as the next operand.  Four warps
    // per row; u and add do not depend on the step before and are fetched ahead of it for the first row.
    const int team = ew >> 2, tt = (ew & 3) * 32 + lane;
    float* red = reinterpret_cast<float*>(c.smem + kWStage + team * 4 * kWStageWarp);
    auto norm_rows = [&](auto per, int splits, auto load_u, auto load_add, const __nv_bfloat16* g, bool enable, float* sum, float* out) {
      constexpr int kPer = decltype(per)::value;
      float uv[CH][4], av[CH][4], gv[CH][4];
#pragma unroll
      for (int k = 0; k < CH; ++k) {
        const int n = 4 * (tt + 128 * k);
#pragma unroll
        for (int e = 0; e < 4; ++e) gv[k][e] = n < d ? gain_at(g, n + e) : 1.f;
      }
      int parity = 0;
      auto fetch = [&](int row) {
#pragma unroll
        for (int k = 0; k < CH; ++k) {
          const int n = 4 * (tt + 128 * k);
          if (n >= d) break;
          load_u(row, n, uv[k]);
          load_add(row, n, av[k]);
        }
      };
      const int row0 = c.rank + team * c.G;
      if (row0 < R) fetch(row0);
      const bool good = epi_all(flag_wait());
      if (!good) return false;
#pragma unroll 1
      for (int row = row0; row < R; row += 2 * c.G) {
        if (row != row0) fetch(row);
        const size_t at = (size_t)(m0 + row) * d;
        float dy[CH][4], ss = 0.f, tu = 0.f;
        float4 pv[CH <= 2 ? CH : 1][kPer];                     // all parts of a row of up to 1024 entries are requested before the first sum
        auto fetch_parts = [&](int k, float4 (&v)[kPer]) {
          const int n = 4 * (tt + 128 * k) < d ? 4 * (tt + 128 * k) : 0;
#pragma unroll
          for (int z = 0; z < kPer; ++z) v[z] = __ldcg(reinterpret_cast<const float4*>(p.partial + (size_t)(z < splits ? z : 0) * rstride + at + n));
        };
        if (CH <= 2) {
#pragma unroll
          for (int k = 0; k < CH; ++k) fetch_parts(k, pv[k < 2 ? k : 0]);
        }
#pragma unroll
        for (int k = 0; k < CH; ++k) {
          const int n = 4 * (tt + 128 * k);
          if (n >= d) break;
          if (CH > 2) fetch_parts(k, pv[0]);
          float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int z = 0; z < kPer; ++z)
            if (z < splits) { acc.x += pv[CH <= 2 ? k : 0][z].x; acc.y += pv[CH <= 2 ? k : 0][z].y; acc.z += pv[CH <= 2 ? k : 0][z].z; acc.w += pv[CH <= 2 ? k : 0][z].w; }
          *reinterpret_cast<float4*>(sum + at + n) = acc;
          dy[k][0] = acc.x; dy[k][1] = acc.y; dy[k][2] = acc.z; dy[k][3] = acc.w;
          if (enable) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              dy[k][e] *= gv[k][e];
              ss = fmaf(uv[k][e], uv[k][e], ss);
              tu = fmaf(dy[k][e], uv[k][e], tu);
            }
          }
        }
        float inv = 1.f, mean = 0.f;
        if (enable) {
          ss = warp_sum(ss); tu = warp_sum(tu);
          if (lane == 0) { red[parity * 8 + (ew & 3)] = ss; red[parity * 8 + 4 + (ew & 3)] = tu; }
          asm volatile("barrier.cta.sync %0, 128;" ::"r"(2 + team) : "memory");
          ss = red[parity * 8] + red[parity * 8 + 1] + red[parity * 8 + 2] + red[parity * 8 + 3];
          tu = red[parity * 8 + 4] + red[parity * 8 + 5] + red[parity * 8 + 6] + red[parity * 8 + 7];
          inv = rsqrtf(ss / d + p.eps); mean = tu * inv / d;
          parity ^= 1;
        }
#pragma unroll
        for (int k = 0; k < CH; ++k) {
          const int n = 4 * (tt + 128 * k);
          if (n >= d) break;
          float r[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) r[e] = av[k][e] + (enable ? inv * (dy[k][e] - uv[k][e] * inv * mean) : dy[k][e]);
          *reinterpret_cast<float4*>(out + at + n) = make_float4(r[0], r[1], r[2], r[3]);
          store_operand4(reinterpret_cast<__nv_bfloat16*>(p.s16) + at + n, r[0] * p.alpha, r[1] * p.alpha, r[2] * p.alpha, r[3] * p.alpha, TERMS, (long long)kWideTermRows * d);
        }
      }
      return true;
    };
    const __nv_bfloat16* Z = reinterpret_cast<const __nv_bfloat16*>(p.z);
    const int t8 = lane & 7;
    // one (sequence, head) per eight lanes, spread over the group's CTAs warp by warp
    const int unit0 = (ew * c.G + c.rank) * 4 + (lane >> 3), unit_stride = 32 * c.G;
    auto col_of = [&](int v, int& b, int& h) { const int w = v < units ? v : 0; b = m0 + w / H; h = w % H; return (size_t)b * d + h * kHeadDim + 8 * t8; };
    // What of a position's attention is off the chain: the leaf's older pairs, by thirds, and the temporary pair (with the first third).  It
    // waits for the products of the next position, whose accumulators the row warps would only wait for.
    auto older_pairs = [&](int i, int third) {
      const int n = i - 1 - p.s0, ja = p.s0 + n * third / 3, jb = p.s0 + n * (third + 1) / 3;
      if (third && ja >= jb) return;
#pragma unroll 1
      for (int v = unit0; v - (lane >> 3) < units; v += unit_stride) {
        int b, h;
        const size_t col = col_of(v, b, h), ri = (size_t)i * rstride + col;
        const bool live = v < units;
        const size_t si = ((size_t)i * p.B + b) * H + h;
        const F8 q = ld8(a.q + ri), dc = ldcg8(p.dc + ri), cc = ld8(a.c + ri);
        const float lse = a.lse[si], slope = a.alibi ? a.alibi[h] * kLog2e : 0.f, D = group_sum(dot8(dc, cc));
        if (third == 0) {
          const F8 kt = ld8(a.kt + ri), vt = ld8(a.vt + ri);
          const float pr = exp2f(group_sum(dot8(q, kt)) * a.scale_log2 - lse);
          const float ds = pr * (group_sum(dot8(dc, vt)) - D) * a.scale;
          F8 o1, o2;
#pragma unroll
          for (int e = 0; e < 8; ++e) { o1.v[e] = ds * q.v[e]; o2.v[e] = pr * dc.v[e]; }
          if (live) { st8(a.dkt + ri, o1); st8(a.dvt + ri, o2); }
        }
#pragma unroll 2
        for (int j = ja; j < jb; ++j) {
          const size_t rj = (size_t)j * rstride + col;
          const F8 kk = ld8(a.k + rj), vv = ld8(a.v + rj);
          F8 gk = ld8(a.dK + rj), gv = ld8(a.dV + rj);
          const float pr = exp2f(group_sum(dot8(q, kk)) * a.scale_log2 - slope * (float)(i - j) - lse);
          const float ds = pr * (group_sum(dot8(dc, vv)) - D) * a.scale;
#pragma unroll
          for (int e = 0; e < 8; ++e) { gk.v[e] = fmaf(ds, q.v[e], gk.v[e]); gv.v[e] = fmaf(pr, dc.v[e], gv.v[e]); }
          if (live) { st8(a.dK + rj, gk); st8(a.dV + rj, gv); }
        }
      }
    };
    bool ok = true;
#pragma unroll 1
    for (int i = p.e0 - 1; i >= p.s0 && ok; --i) {
      const size_t od = (size_t)i * rstride, of = (size_t)i * p.B * p.dff;
      if (c.rank < active_of(B_KV)) {
        ok = finish(plain_product(p.st[0], p.partial), B_KV);
        if (!ok) break;
      }
      if (c.rank < active_of(B_RZ)) {
        auto rows = [&](auto per) {
          return norm_rows(per, p.st[0].splits,
                       [&](int row, int n, float (&v)[4]) { reinterpret_cast<const Vec4<__nv_bfloat16>*>(Z + (size_t)(m0 + row) * p.z_bs + (size_t)i * p.z_ts + n)->to_float(v); },
                       [&](int row, int n, float (&v)[4]) { reinterpret_cast<const Vec4<float>*>(p.dz + (size_t)(m0 + row) * p.dz_bs + (size_t)i * p.dz_ts + n)->to_float(v); },
                       reinterpret_cast<const __nv_bfloat16*>(p.g_kv), p.z_norm != 0, p.dr + od, p.Gz + od);
        };
        ok = p.st[0].splits > 4 ? rows(std::integral_constant<int, 8>()) : rows(std::integral_constant<int, 4>());
        ok = finish(ok, B_RZ);
        if (!ok) break;
      }
      if (i + 1 < p.e0) older_pairs(i + 1, 0);
      if (c.rank < active_of(B_DOWN)) {
        // dpre = (alpha Gz W_down) GELU'(act)
        bool good = flag_wait();
        const WideStage& st = p.st[1];
#pragma unroll 1
        for (int job = c.rank; job < st.tiles; job += c.G) {
          const int n0 = job * st.bn;
          const int cols = st.bn >> 1;                          // 32 or 64 of this warp; GELU' is ready before the accumulators are
          float4 xv[2][kIter];
#pragma unroll
          for (int q = 0; q < 2; ++q) {
#pragma unroll
            for (int k = 0; k < kIter; ++k) {
              const int rr = row_of0 + row_base + 4 * k + (lane >> 3);
              if (32 * q < cols) xv[q][k] = *reinterpret_cast<const float4*>(p.act + of + (size_t)(m0 + (rr < R ? rr : 0)) * p.dff + n0 + half * cols + 32 * q + 4 * (lane & 7));
            }
          }
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            if (32 * q >= cols) break;
#pragma unroll
            for (int k = 0; k < kIter; ++k)
              xv[q][k] = make_float4(gelu_grad_wide(xv[q][k].x), gelu_grad_wide(xv[q][k].y), gelu_grad_wide(xv[q][k].z), gelu_grad_wide(xv[q][k].w));
          }
          if (good) good = acc_wait();
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            if (32 * q >= cols) break;
            const int cc = half * cols + 32 * q;
            const bool done = staged(good, cc, [&](int k, int rr, int col, const float4& v) {
              const float4 x = xv[q][k];
              const float4 o = make_float4(v.x * x.x, v.y * x.y, v.z * x.z, v.w * x.w);
              if (rr < R) {
                const size_t at = (size_t)(m0 + rr) * p.dff + n0 + cc + col;
                *reinterpret_cast<float4*>(p.dpre + of + at) = o;
                store_operand4(reinterpret_cast<__nv_bfloat16*>(p.p16) + at, o.x, o.y, o.z, o.w, TERMS, (long long)kWideTermRows * p.dff);
              }
            });
            good = good && done;
          }
          if (!good) break;
          acc_done();
        }
        ok = finish(good, B_DOWN);
        if (!ok) break;
      }
      if (i + 1 < p.e0) older_pairs(i + 1, 1);
      if (c.rank < active_of(B_UP)) {
        ok = finish(plain_product(p.st[2], p.partial), B_UP);
        if (!ok) break;
      }
      if (c.rank < active_of(B_RH)) {
        auto rows = [&](auto per) {
          return norm_rows(per, p.st[2].splits,
                       [&](int row, int n, float (&v)[4]) { reinterpret_cast<const Vec4<float>*>(p.h + od + (size_t)(m0 + row) * d + n)->to_float(v); },
                       [&](int row, int n, float (&v)[4]) { reinterpret_cast<const Vec4<float>*>(p.Gz + od + (size_t)(m0 + row) * d + n)->to_float(v); },     // this thread's own
                       reinterpret_cast<const __nv_bfloat16*>(p.g_mlp), p.pre != 0, p.du + od, p.dh + od);
        };
        ok = p.st[2].splits > 4 ? rows(std::integral_constant<int, 8>()) : rows(std::integral_constant<int, 4>());
        ok = finish(ok, B_RH);
        if (!ok) break;
      }
      if (i + 1 < p.e0) older_pairs(i + 1, 2);
      if (c.rank < active_of(B_OUT)) {
        ok = finish(plain_product(p.st[3], p.dc + od), B_OUT);
        if (!ok) break;
      }
      if (c.rank < active_of(B_ATTN)) {
        bool waited = false;
#pragma unroll 1
        for (int v = unit0; v - (lane >> 3) < units && ok; v += unit_stride) {
          int b, h;
          const size_t col = col_of(v, b, h), ri = od + col, rj = ri - rstride;
          const bool live = v < units, newest = i > p.s0;
          const size_t si = ((size_t)i * p.B + b) * H + h;
          const F8 q = ld8(a.q + ri), cc = ld8(a.c + ri);
          const float lse = a.lse[si], slope = a.alibi ? a.alibi[h] * kLog2e : 0.f;
          F8 kk, vv, gk, gv, kr;
          if (newest) { kk = ld8(a.k + rj); vv = ld8(a.v + rj); gk = ld8(a.dK + rj); gv = ld8(a.dV + rj); kr = ld8(wp.kraw + rj); }
          if (!waited) { ok = flag_wait(); waited = true; }
          if (!ok) break;
          const F8 dc = ldcg8(p.dc + ri);
          const float D = group_sum(dot8(dc, cc));
          if (newest) {
            const float pr = exp2f(group_sum(dot8(q, kk)) * a.scale_log2 - slope - lse);
            const float ds = pr * (group_sum(dot8(dc, vv)) - D) * a.scale;
#pragma unroll
            for (int e = 0; e < 8; ++e) { gk.v[e] = fmaf(ds, q.v[e], gk.v[e]); gv.v[e] = fmaf(pr, dc.v[e], gv.v[e]); }
            if (live) { st8(a.dK + rj, gk); st8(a.dV + rj, gv); }
            pair_operand(gk, gv, kr, wp, b, d, h, t8, wp.dkraw + rj, live);
          }
          if (live && t8 == 0) a.D[si] = D;
        }
        if (!waited) ok = flag_wait();
        ok = finish(ok, B_ATTN);
        if (!ok) break;
      }
    }
    if (ok) older_pairs(p.s0, 0);                              // (the first position's temporary pair)
  }
  wide_teardown(tmem, warp);
}
}  // namespace

// Of the reverse loop: 0, or the number of groups.  A row of more than 4096 entries would not fit the registers of its four warps.
int wide_backward_groups(int B, int d, int dff) { return d <= 4096 ? wide_loop_groups(B, d, dff) : 0; }

cudaError_t wide_backward_launch(WideBwdParams p, const AttnBufs& a, const WidePair& wp, cudaStream_t s) {
  const int groups = wide_backward_groups(p.B, p.d, p.dff);
  if (!groups) return cudaErrorInvalidValue;
  p.R = ceil_div(p.B, groups); p.G = kB200Sms / groups;
  const int box = p.terms == 3 ? 3 * kWideTermRows : (p.R + 7) / 8 * 8, rows = p.terms == 3 ? box : p.B;
  p.a_bytes = box * 128;
  p.st[0] = stage_split(p.d, 2 * p.d, p.G, p.a_bytes);
  p.st[1] = stage_whole(p.dff, p.d, p.G, p.a_bytes, 128);
  p.st[2] = stage_split(p.d, p.dff, p.G, p.a_bytes);
  p.st[3] = stage_whole(p.d, p.d, p.G, p.a_bytes, 128);
  WideBwdMaps m;
  const void *A[4] = {wp.op, p.s16, p.p16, p.s16}, *W[4] = {p.wkvT, p.wdnT, p.wupT, p.woT};
  const int K[4] = {2 * p.d, p.d, p.dff, p.d}, N[4] = {p.d, p.dff, p.d, p.d};
  for (int i = 0; i < 4; ++i)
    if (!map_blocks(&m.a[i], A[i], rows, K[i], box) || !map_blocks(&m.w[i], W[i], N[i], K[i], p.st[i].bn)) return cudaErrorInvalidValue;
  const void* fn = p.terms == 3 ? (p.d <= 1024 ? reinterpret_cast<const void*>(&wide_backward_kernel<2, 3>) : reinterpret_cast<const void*>(&wide_backward_kernel<8, 3>))
                                : (p.d <= 1024 ? reinterpret_cast<const void*>(&wide_backward_kernel<2, 1>) : reinterpret_cast<const void*>(&wide_backward_kernel<8, 1>));
  const int smem = (int)kWTotal + 1024;
  cudaError_t e = ensure_dynamic_smem(fn, smem);
  if (e != cudaSuccess) return e;
  void* args[] = {(void*)&m, (void*)&p, (void*)&a, (void*)&wp};
  return cudaLaunchCooperativeKernel(fn, dim3(groups * p.G), dim3(kWThreads), args, smem, s);
}

}  // namespace rt
