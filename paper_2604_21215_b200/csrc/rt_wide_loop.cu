// Token loop of wide batches (up to 128 sequences per group of SMs), one cooperative launch per leaf, bf16.
//
// A token step of B sequences is a chain of dense products over B rows.  As separate launches (rt_recompute.cu, rt_prepass_tc.cu,
// rt_tile.cu) a position of a layer of width 1024 is seven or eight launches of 5 to 8 us each, of which two thirds are launch, fill and
// drain: every launch begins with an empty pipeline and fetches its weights only then.  Here the chain runs inside one kernel:
//   - the batch is cut into groups of at most 128 sequences (one row tile of the tensor cores); a group of 148 / groups SMs runs its
//     positions on its own (sequences are independent), so steps meet at a barrier of that group only;
//   - one CTA per SM, three roles: warp 0 fetches operands by TMA, warp 1 issues tcgen05.mma, eight warps read the accumulators and do the
//     row-wise work (attention, sums of split products);
//   - the weights of the next product do not depend on the step before it: warp 0 fetches them while it waits, and only the operand rows
//     (at most 128 KB to 256 KB per CTA, at 145 GB/s per SM) and the barrier stay on the chain.
// RMS norms need whole rows, which no CTA owns: the product's epilogue leaves h * gain in bf16 and the sums of squares of its columns, and
// the next product scales its accumulator rows by 1 / rms.  The down projection contracts over d_ff: it runs in up to eight parts whose sums
// meet in a row step.
//
// Exchange: data through global memory (L2), a counter per step and group (release by one thread after a barrier of the CTA's row warps,
// acquire and a proxy fence by the warp that then fetches).  Every wait is bounded (2 s).
//
// Measured per position at d = 1024, d_ff = 4096, against the launches: B = 96 27.6 us (42), B = 200 (d = 768) 27 (50), B = 512 38 (57).  A step
// is about 1 us from the last count to the first fetch, 2 to 5 us until the accumulators are complete (operand rows and weights at 145 GB/s
// per SM, about 1.2 us of latency), 1 to 2.5 us of row work, 0.7 us for the release.
#include <type_traits>

#include "rt_wide.cuh"

namespace rt {

namespace {
// ---- attention of one (sequence, head) on eight lanes: the row's state (the pre-pass and the tiles before this leaf) and the leaf's keys
struct WideAttn { uint4 q; float o[8], m, l; unsigned col; };      // q in bf16; col: offset of the eight entries within a position's rows [B, d]
// the keys [ka, kb) of two units, four keys at a time
__device__ __forceinline__ void wide_attn_keys(WideAttn (&a)[2], const __nv_bfloat16* K, const __nv_bfloat16* V, size_t rstride, int ka, int kb, int t, float scale_log2, const float* alibi, int d) {
  float slope[2] = {0.f, 0.f};
  if (alibi) { slope[0] = alibi[a[0].col % d / kHeadDim] * kLog2e; slope[1] = alibi[a[1].col % d / kHeadDim] * kLog2e; }
#pragma unroll 1
  for (int j0 = ka; j0 < kb; j0 += 4) {
    uint4 kw[2][4], vw[2][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const size_t at = (size_t)(j0 + e < kb ? j0 + e : kb - 1) * rstride;
#pragma unroll
      for (int i = 0; i < 2; ++i) { kw[i][e] = ldcg16(K + at + a[i].col); vw[i][e] = ldcg16(V + at + a[i].col); }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      float s[4], qf[8], m_new = a[i].m;
      unpack8(a[i].q, qf);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float kf[8], x = 0.f;
        unpack8(kw[i][e], kf);
#pragma unroll
        for (int k = 0; k < 8; ++k) x = fmaf(qf[k], kf[k], x);
        x = sum8(x);
        s[e] = j0 + e < kb ? x * scale_log2 - slope[i] * (float)(t - (j0 + e)) : -INFINITY;
        m_new = fmaxf(m_new, s[e]);
      }
      const float corr = exp2f(a[i].m - m_new);
      a[i].l *= corr; a[i].m = m_new;
#pragma unroll
      for (int k = 0; k < 8; ++k) a[i].o[k] *= corr;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float pj = exp2f(s[e] - m_new);
        float vf[8];
        unpack8(vw[i][e], vf);
        a[i].l += pj;
#pragma unroll
        for (int k = 0; k < 8; ++k) a[i].o[k] = fmaf(pj, vf[k], a[i].o[k]);
      }
    }
  }
}
// one key whose rows have been fetched
__device__ __forceinline__ void wide_attn_one(WideAttn& a, const uint4& kw, const uint4& vw, float scale_log2, float slope) {
  float kf[8], vf[8], qf[8], x = 0.f;
  unpack8(kw, kf); unpack8(vw, vf); unpack8(a.q, qf);
#pragma unroll
  for (int i = 0; i < 8; ++i) x = fmaf(qf[i], kf[i], x);
  const float s = sum8(x) * scale_log2 - slope, m_new = fmaxf(a.m, s);
  const float corr = exp2f(a.m - m_new), pj = exp2f(s - m_new);
  a.m = m_new; a.l = a.l * corr + pj;
#pragma unroll
  for (int i = 0; i < 8; ++i) a.o[i] = fmaf(pj, vf[i], a.o[i] * corr);
}

// ---- forward ------------------------------------------------------------------------------------------------
enum { F_ATTN = 0, F_OUT = 1, F_UP = 2, F_DOWN = 3, F_Z = 4, F_KV = 5, F_STEPS = 6 };

// The products in the order of the chain (indices of WideFwdParams::st): W_o, W_up, W_down, W_k | W_v; the last map is W_v's.
struct WideFwdMaps { CUtensorMap a[4], w[5]; };

__global__ void __launch_bounds__(kWThreads, 1) wide_forward_kernel(const __grid_constant__ WideFwdMaps maps, const __grid_constant__ WideFwdParams p) {
  extern __shared__ unsigned char smem_raw[];
  WideCta c;
  c.smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  c.sbase = smem_u32(c.smem);
  c.s_abort = reinterpret_cast<volatile int*>(c.smem + kWAbort);
  c.sync = p.sync;
  c.G = p.G;
  const int group = blockIdx.x / p.G;
  c.rank = blockIdx.x % p.G;
  c.arank = p.G - 1 - c.rank;
  c.counters = p.counters + group * kWMaxSteps * kWCounterStride;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int m0 = group * p.R, R = p.B - m0 < p.R ? p.B - m0 : p.R;
  volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(c.smem + kWTmem);
  wide_setup(c, tid, warp);
  const uint32_t tmem = *s_tmem, a_bytes = (uint32_t)p.a_bytes;

  const int d = p.d, H = p.H, chunks = d >> 7;
  auto active_of = [&](int step) {                             // CTAs of the group that have work in a step
    if (step == F_ATTN) return wide_active_rows(R * H, 64, p.G);
    if (step == F_Z) return wide_active_rows(R * chunks, 8, p.G);
    return wide_active(p.st[step < F_Z ? step - 1 : 3], p.G);
  };

  if (warp == 0) {
    // ---------------- operand fetches and the group's barrier ----------------
    WideFetch f = {0u, 0u};
    bool ok = true;
#pragma unroll 1
    for (int t = p.t0; t < p.t1 && ok; ++t) {
      const unsigned n = p.steps + (unsigned)(t - p.t0);                     // positions done before this one
      int product = 0;
#pragma unroll 1
      for (int step = 0; step < F_STEPS && ok; ++step) {
        const bool rows = step == F_ATTN || step == F_Z;
        const int mine = step == F_ATTN ? c.arank : c.rank;
        auto wait = [&]() {
          bool r = true;
          if (step == F_ATTN) { if (t > p.t0) r = c.poll(F_KV, n * (unsigned)active_of(F_KV)); }
          else r = c.poll(step - 1, (n + 1) * (unsigned)active_of(step - 1));
          if (lane == 0 && r) mbar_arrive(c.flag());
          __syncwarp();
          return r;
        };
        if (mine < active_of(step)) {
          if (rows) ok = wait();
          else ok = wide_fetch(c, f, p.st[product], &maps.a[product], &maps.w[product], step == F_KV ? &maps.w[4] : nullptr, m0, a_bytes, wait);
        }
        if (!rows) ++product;
      }
    }
  } else if (warp == 1) {
    // ---------------- tensor cores ----------------
    WideIssue w = {0u, 0};
    bool ok = true;
#pragma unroll 1
    for (int t = p.t0; t < p.t1 && ok; ++t)
#pragma unroll 1
      for (int product = 0; product < 4 && ok; ++product) ok = wide_issue(c, w, p.st[product], a_bytes, tmem);
  } else {
    // ---------------- row work: eight warps, a warp reads the 32 TMEM lanes of its quadrant, two warps share a quadrant's columns ----------------
    const int ew = warp - 2, quad = warp & 3, half = ew >> 2;
    const int row = quad * 32 + lane, m = m0 + row;
    const bool live = row < R;
    const uint32_t t_row = tmem + ((uint32_t)(quad * 32) << 16);
    const bool pre = (p.norm_flags & RT_NORM_PRE) != 0, znorm = pre && !(p.norm_flags & RT_NORM_SKIP_Z), qkn = (p.norm_flags & RT_NORM_QK) != 0;
    const __nv_bfloat16 *g_mlp = reinterpret_cast<const __nv_bfloat16*>(p.g_mlp), *g_kv = reinterpret_cast<const __nv_bfloat16*>(p.g_kv), *g_k = reinterpret_cast<const __nv_bfloat16*>(p.g_k);
    const __nv_bfloat16 *X = reinterpret_cast<const __nv_bfloat16*>(p.x), *Q = reinterpret_cast<const __nv_bfloat16*>(p.q);
    __nv_bfloat16 *Z = reinterpret_cast<__nv_bfloat16*>(p.z), *Kc = reinterpret_cast<__nv_bfloat16*>(p.k_cache), *Vc = reinterpret_cast<__nv_bfloat16*>(p.v_cache);
    const size_t rstride = (size_t)p.B * d;
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
    auto finish = [&](bool ok, int step) {                     // this CTA's part of a step is written
      ok = epi_all(ok);
      if (tid == 64 && ok) { red_release_add_u32(c.counters + step * kWCounterStride, 1u); }
      return ok;
    };
    // 1 / rms of this thread's row from the sums of squares that the step before left ([part][B])
    auto row_scale = [&](const float* ssq, int parts, bool on) {
      if (!on || !live) return 1.0f;
      float sum = 0.f;
      const float* a = ssq + m;
#pragma unroll 1
      for (int i0 = 0; i0 < parts; i0 += 16) {
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = i0 + i < parts ? __ldcg(a + (size_t)(i0 + i) * p.B) : 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) sum += v[i];
      }
      return rsqrtf(sum / (float)d + p.eps);
    };
    float* stage = reinterpret_cast<float*>(c.smem + kWStage + ew * kWStageWarp);
    // this warp's half of an accumulator of bn columns, entry(value) by the lane of the row, then f(row of the quadrant, column, values) by every lane
    auto blocks = [&](int bn, auto entry, auto f) {
#pragma unroll 1
      for (int cc = half * (bn >> 1); cc < (half + 1) * (bn >> 1); cc += 32) {
        wide_stage(stage, t_row + (uint32_t)((jobs & 1) * kWBuf + cc), lane, entry);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = 4 * i + (lane >> 3), col = 4 * (lane & 7);
          f(r, cc + col, *reinterpret_cast<const float4*>(stage + r * kWStagePitch + col));
        }
      }
    };
    // Attention: eight lanes per (sequence, head), two of these at a time per group of lanes.  The state of the row and the leaf's keys but the
    // newest are taken in while the four products of the position before are under way, a quarter of the keys in front of each.
    const int units = R * H, unit0 = c.arank * 64 + ew * 8 + (lane >> 3);
    WideAttn at[2];
    auto attn_begin = [&](int u0, int t) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int u = u0 + 4 * i < units ? u0 + 4 * i : 0, b = m0 + u / H, h = u % H;
        const size_t sidx = (size_t)t * p.B + b;
        at[i].col = (unsigned)(b * d + h * kHeadDim + 8 * (lane & 7));
        const size_t row = (size_t)t * rstride + at[i].col;
        at[i].q = *reinterpret_cast<const uint4*>(Q + row);
        const float4 o0 = *reinterpret_cast<const float4*>(p.st_o + row), o1 = *reinterpret_cast<const float4*>(p.st_o + row + 4);
        at[i].o[0] = o0.x; at[i].o[1] = o0.y; at[i].o[2] = o0.z; at[i].o[3] = o0.w; at[i].o[4] = o1.x; at[i].o[5] = o1.y; at[i].o[6] = o1.z; at[i].o[7] = o1.w;
        at[i].m = p.st_m[sidx * H + h]; at[i].l = p.st_l[sidx * H + h];
      }
    };
    const bool attends = c.arank < active_of(F_ATTN);
    if (attends) attn_begin(unit0, p.t0);
    bool ok = true;
#pragma unroll 1
    for (int t = p.t0; t < p.t1 && ok; ++t) {
#pragma unroll 1
    for (int step = 0; step < F_STEPS; ++step) {
      if (attends && t + 1 < p.t1 && step != F_ATTN && step != F_Z) {
        const int product = step < F_Z ? step - 1 : 3, per = ((t - p.t0 + 3) / 4 + 3) / 4 * 4;     // whole batches of four keys
        if (product == 0) attn_begin(unit0, t + 1);
        const int ka = p.t0 + product * per, kb = ka + per < t ? ka + per : t;
        wide_attn_keys(at, Kc, Vc, rstride, ka, kb, t + 1, p.scale_log2, p.alibi, d);
      }
      if (step == F_ATTN && attends) {
        const int per_round = 64 * c.G;
        bool waited = false;
#pragma unroll 1
        for (int u0 = unit0; u0 - (lane >> 3) < units && ok; u0 += per_round) {
          if (u0 != unit0) { attn_begin(u0, t); wide_attn_keys(at, Kc, Vc, rstride, p.t0, t - 1, t, p.scale_log2, p.alibi, d); }
          if (!waited) { ok = flag_wait(); waited = true; }
          if (!ok) break;
          if (t > p.t0) {
            uint4 kn[2], vn[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) { kn[i] = ldcg16(Kc + (size_t)(t - 1) * rstride + at[i].col); vn[i] = ldcg16(Vc + (size_t)(t - 1) * rstride + at[i].col); }
#pragma unroll
            for (int i = 0; i < 2; ++i) wide_attn_one(at[i], kn[i], vn[i], p.scale_log2, p.alibi ? p.alibi[at[i].col % d / kHeadDim] * kLog2e : 0.f);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const float il = 1.0f / at[i].l;
            if (u0 + 4 * i < units)
              *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(p.c16) + at[i].col) =
                  make_uint4(pack2(at[i].o[0] * il, at[i].o[1] * il), pack2(at[i].o[2] * il, at[i].o[3] * il), pack2(at[i].o[4] * il, at[i].o[5] * il), pack2(at[i].o[6] * il, at[i].o[7] * il));
          }
        }
        if (!waited) ok = flag_wait();                         // (a warp without units)
        ok = finish(ok, F_ATTN);
        if (!ok) break;
      }
      if (step == F_OUT && c.rank < active_of(F_OUT)) {
        // h = x + alpha c W_o;  u = bf16(h g), sums of squares of h
        bool good = flag_wait();
        const int bn = p.st[0].bn;
#pragma unroll 1
        for (int job = c.rank; job < p.st[0].tiles; job += c.G) {
          const int n0 = job * bn;
          uint2 xw[8];                                         // x of the first 32 columns: fetched before the accumulators are there
          auto fetch_x = [&](int cc) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int rr = quad * 32 + 4 * i + (lane >> 3);
              xw[i] = *reinterpret_cast<const uint2*>(X + (size_t)(m0 + (rr < R ? rr : 0)) * p.x_bs + (size_t)t * p.x_ts + n0 + cc + 4 * (lane & 7));
            }
          };
          fetch_x(half * (bn >> 1));
          if (!good || !(good = acc_wait())) break;
          float sums[8] = {};
#pragma unroll 1
          for (int cc = half * (bn >> 1); cc < (half + 1) * (bn >> 1); cc += 32) {
            if (cc != half * (bn >> 1)) fetch_x(cc);
            const int n = n0 + cc + 4 * (lane & 7);
            float g0 = 1.f, g1 = 1.f, g2 = 1.f, g3 = 1.f;
            if (pre && g_mlp) {
              const uint2 gw = *reinterpret_cast<const uint2*>(g_mlp + n);
              g0 = __uint_as_float(gw.x << 16); g1 = __uint_as_float(gw.x & 0xffff0000u); g2 = __uint_as_float(gw.y << 16); g3 = __uint_as_float(gw.y & 0xffff0000u);
            }
            wide_stage(stage, t_row + (uint32_t)((jobs & 1) * kWBuf + cc), lane, [](float v) { return v; });
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int r = 4 * i + (lane >> 3);
              const float4 a = *reinterpret_cast<const float4*>(stage + r * kWStagePitch + 4 * (lane & 7));
              const float h0 = __uint_as_float(xw[i].x << 16) + p.alpha * a.x, h1 = __uint_as_float(xw[i].x & 0xffff0000u) + p.alpha * a.y,
                          h2 = __uint_as_float(xw[i].y << 16) + p.alpha * a.z, h3 = __uint_as_float(xw[i].y & 0xffff0000u) + p.alpha * a.w;
              sums[i] = fmaf(h0, h0, fmaf(h1, h1, fmaf(h2, h2, fmaf(h3, h3, sums[i]))));
              if (quad * 32 + r < R) {
                const size_t at = (size_t)(m0 + quad * 32 + r) * d + n;
                *reinterpret_cast<float4*>(p.h + at) = make_float4(h0, h1, h2, h3);
                *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.u16) + at) = make_uint2(pack2(h0 * g0, h1 * g1), pack2(h2 * g2, h3 * g3));
              }
            }
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) {                        // the sum of squares of a row over this warp's columns
            const float v = sum8(sums[i]);
            const int rr = quad * 32 + 4 * i + (lane >> 3);
            if ((lane & 7) == 0 && rr < R) p.ssq_h[(size_t)(2 * job + half) * p.B + m0 + rr] = v;
          }
          acc_done();
        }
        ok = finish(good, F_OUT);
        if (!ok) break;
      }
      if (step == F_UP && c.rank < active_of(F_UP)) {
        // g = GELU(u W_up / rms(h))
        bool good = flag_wait();
        const float inv = good ? row_scale(p.ssq_h, p.st[0].tiles * 2, pre) : 1.f;
        const int bn = p.st[1].bn;
#pragma unroll 1
        for (int job = c.rank; job < p.st[1].tiles; job += c.G) {
          if (!good || !(good = acc_wait())) break;
          blocks(bn, [&](float v) { return gelu_wide(v * inv); }, [&](int r, int col, const float4& a) {
            if (quad * 32 + r < R)
              *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.g16) + (size_t)(m0 + quad * 32 + r) * p.dff + job * bn + col) = make_uint2(pack2(a.x, a.y), pack2(a.z, a.w));
          });
          acc_done();
        }
        ok = finish(good, F_UP);
        if (!ok) break;
      }
      if (step == F_DOWN && c.rank < active_of(F_DOWN)) {
        // a part of g W_down
        bool good = flag_wait();
        const int bn = p.st[2].bn;
#pragma unroll 1
        for (int job = c.rank; job < p.st[2].tiles * p.st[2].splits; job += c.G) {
          const int n0 = (job % p.st[2].tiles) * bn, split = job / p.st[2].tiles;
          if (!good || !(good = acc_wait())) break;
          blocks(bn, [](float v) { return v; }, [&](int r, int col, const float4& a) {
            if (quad * 32 + r < R) *reinterpret_cast<float4*>(p.partial + ((size_t)split * p.B + m0 + quad * 32 + r) * d + n0 + col) = a;
          });
          acc_done();
        }
        ok = finish(good, F_DOWN);
        if (!ok) break;
      }
      if (step == F_Z && c.rank < active_of(F_Z)) {
        // z = h + alpha g W_down;  r = bf16(z g), sums of squares of z: a warp per row and 128 columns
        const int total = R * chunks, stride = c.G * 8, splits = p.st[2].splits;
        const bool ahead = c.rank < active_of(F_UP) || c.rank < active_of(F_DOWN);      // such a CTA has seen that h is complete
        bool good = true, waited = false;
        // ROWS units with PER parts each are fetched together
        auto units_of = [&](auto rows, auto per) {
          constexpr int kRows = decltype(rows)::value, kPer = decltype(per)::value;
#pragma unroll 1
          for (int u0 = c.rank * 8 + ew; u0 < total; u0 += kRows * stride) {
            int b[kRows], col[kRows];
            float4 hv[kRows], pv[kRows][kPer];
#pragma unroll
            for (int k = 0; k < kRows; ++k) {
              const int u = u0 + k * stride < total ? u0 + k * stride : u0;
              b[k] = m0 + u / chunks; col[k] = (u % chunks) * 128 + 4 * lane;
            }
            auto fetch_h = [&]() {
#pragma unroll
              for (int k = 0; k < kRows; ++k) hv[k] = __ldcg(reinterpret_cast<const float4*>(p.h + (size_t)b[k] * d + col[k]));
            };
            if (ahead || waited) fetch_h();
            if (!waited) {
              good = flag_wait();
              waited = true;
              if (!good) break;
              if (!ahead) fetch_h();
            }
#pragma unroll
            for (int k = 0; k < kRows; ++k)
#pragma unroll
              for (int z = 0; z < kPer; ++z) pv[k][z] = __ldcg(reinterpret_cast<const float4*>(p.partial + ((size_t)(z < splits ? z : 0) * p.B + b[k]) * d + col[k]));
#pragma unroll
            for (int k = 0; k < kRows; ++k) {
              if (u0 + k * stride >= total) break;
              float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
              for (int z = 0; z < kPer; ++z)
                if (z < splits) { acc.x += pv[k][z].x; acc.y += pv[k][z].y; acc.z += pv[k][z].z; acc.w += pv[k][z].w; }
              float v[4] = {hv[k].x + p.alpha * acc.x, hv[k].y + p.alpha * acc.y, hv[k].z + p.alpha * acc.z, hv[k].w + p.alpha * acc.w};
              float ss = 0.f;
#pragma unroll
              for (int i = 0; i < 4; ++i) { v[i] = round_T<__nv_bfloat16>(v[i]); ss = fmaf(v[i], v[i], ss); }    // the pair comes from the stored (rounded) z
              *reinterpret_cast<uint2*>(Z + (size_t)b[k] * p.z_bs + (size_t)t * p.z_ts + col[k]) = make_uint2(pack2(v[0], v[1]), pack2(v[2], v[3]));
              ss = warp_sum(ss);
              if (lane == 0) p.ssq_z[(size_t)(col[k] >> 7) * p.B + b[k]] = ss;
              if (znorm && g_kv) {
                const uint2 gw = *reinterpret_cast<const uint2*>(g_kv + col[k]);
                v[0] *= __uint_as_float(gw.x << 16); v[1] *= __uint_as_float(gw.x & 0xffff0000u); v[2] *= __uint_as_float(gw.y << 16); v[3] *= __uint_as_float(gw.y & 0xffff0000u);
              }
              *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.r16) + (size_t)b[k] * d + col[k]) = make_uint2(pack2(v[0], v[1]), pack2(v[2], v[3]));
            }
          }
        };
        if (splits > 4) units_of(std::integral_constant<int, 1>(), std::integral_constant<int, 8>());
        else units_of(std::integral_constant<int, 2>(), std::integral_constant<int, 4>());
        if (!waited) good = flag_wait();                       // (a warp without units)
        ok = finish(good, F_Z);
        if (!ok) break;
      }
      if (step == F_KV && c.rank < active_of(F_KV)) {
        // k = qkRMS(r W_k / rms(z)), v = r W_v / rms(z): a tile is one head
        bool good = flag_wait();
        const float inv = good ? row_scale(p.ssq_z, chunks, znorm) : 1.f;
        const int heads = d / kHeadDim;
#pragma unroll 1
        for (int job = c.rank; job < p.st[3].tiles; job += c.G) {
          if (!good || !(good = acc_wait())) break;
          const bool is_k = job < heads;
          const int col = (is_k ? job : job - heads) * kHeadDim;
          float v[32], ss = 0.f;
          {
            uint32_t w[32];
            tc_ld32(t_row + (uint32_t)((jobs & 1) * kWBuf + half * 32), w);
            tc_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i) { v[i] = __uint_as_float(w[i]) * inv; ss = fmaf(v[i], v[i], ss); }
          }
          if (is_k && qkn) {
            uint32_t w[32];
            tc_ld32(t_row + (uint32_t)((jobs & 1) * kWBuf + (half ^ 1) * 32), w);
            tc_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i) { const float x = __uint_as_float(w[i]) * inv; ss = fmaf(x, x, ss); }
          }
          acc_done();
          const float rs = is_k && qkn ? rsqrtf(ss * (1.0f / kHeadDim) + p.eps) : 1.0f;
          const int cc = col + half * 32;
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 8; ++i) *reinterpret_cast<float4*>(stage + lane * kWStagePitch + 4 * i) = make_float4(v[4 * i] * rs, v[4 * i + 1] * rs, v[4 * i + 2] * rs, v[4 * i + 3] * rs);
          __syncwarp();
          float g[4] = {1.f, 1.f, 1.f, 1.f};
          if (is_k && qkn && g_k) {
#pragma unroll
            for (int i = 0; i < 4; ++i) g[i] = __bfloat162float(g_k[cc + 4 * (lane & 7) + i]);
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int r = 4 * i + (lane >> 3), rr = quad * 32 + r;
            const float4 o = *reinterpret_cast<const float4*>(stage + r * kWStagePitch + 4 * (lane & 7));
            if (rr < R)
              *reinterpret_cast<uint2*>((is_k ? Kc : Vc) + (size_t)t * rstride + (size_t)(m0 + rr) * d + cc + 4 * (lane & 7)) = make_uint2(pack2(o.x * g[0], o.y * g[1]), pack2(o.z * g[2], o.w * g[3]));
          }
        }
        ok = finish(good, F_KV);
      }
    }
    }
  }
  wide_teardown(tmem, warp);
}

}  // namespace

// Groups of at most 128 sequences; beyond kWideGroupsMax of them (16 SMs each or fewer) the products are long enough for launches of their own.
int wide_loop_groups(int B, int d, int dff) {
  const int groups = ceil_div(B, kBM);
  return d % 128 == 0 && dff % 128 == 0 && groups <= kWideGroupsMax ? groups : 0;
}
size_t wide_counter_bytes(int B) { return (size_t)ceil_div(B, kBM) * kWMaxSteps * kWCounterStride * sizeof(unsigned); }
int wide_ssq_floats(int d) { return d / 32 + d / 128; }        // per sequence: parts of ssq_h (at most d / 32), of ssq_z

cudaError_t wide_forward_launch(WideFwdParams p, cudaStream_t s) {
  const int groups = wide_loop_groups(p.B, p.d, p.dff);
  if (!groups) return cudaErrorInvalidValue;
  p.R = ceil_div(p.B, groups); p.G = kB200Sms / groups;
  const int box = (p.R + 7) / 8 * 8;
  p.a_bytes = box * 128;
  p.st[0] = stage_whole(p.d, p.d, p.G, p.a_bytes, 128);
  p.st[1] = stage_whole(p.dff, p.d, p.G, p.a_bytes, 128);
  p.st[2] = stage_split(p.d, p.dff, p.G, p.a_bytes);
  p.st[3] = stage_whole(2 * p.d, p.d, p.G, p.a_bytes, 64);               // a tile is one head
  p.ssq_z = p.ssq_h + (size_t)(p.d / 32) * p.B;
  WideFwdMaps m;
  const void *A[4] = {p.c16, p.u16, p.g16, p.r16}, *W[5] = {p.w_o, p.w_up, p.w_down, p.w_k, p.w_v};
  const int K[5] = {p.d, p.d, p.dff, p.d, p.d}, N[5] = {p.d, p.dff, p.d, p.d, p.d};
  bool ok = true;
  for (int i = 0; i < 5; ++i) {
    const WideStage& st = p.st[i < 4 ? i : 3];
    if (i < 4) ok = ok && map_blocks(&m.a[i], A[i], p.B, K[i], box);
    ok = ok && map_blocks(&m.w[i], W[i], N[i], K[i], st.bn);
  }
  if (!ok)
    return cudaErrorInvalidValue;
  const void* fn = reinterpret_cast<const void*>(&wide_forward_kernel);
  const int smem = (int)kWTotal + 1024;
  cudaError_t e = ensure_dynamic_smem(fn, smem);
  if (e != cudaSuccess) return e;
  void* args[] = {(void*)&m, (void*)&p};
  return cudaLaunchCooperativeKernel(fn, dim3(groups * p.G), dim3(kWThreads), args, smem, s);
}

}  // namespace rt
