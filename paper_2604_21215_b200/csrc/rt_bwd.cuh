// Attention terms of the backward pass, shared by its all-pairs kernels and the loop of wide batches.
#pragma once
#include "rt_kernels.h"
#include "rt_common.cuh"

namespace rt {

struct AttnBufs {
  const float *q, *k, *v, *kt, *vt;        // position-major [rows, d]
  float *lse, *D;                          // [rows, H]: log2-sum-exp of the logits (log2 units), <dc, c> per head
  float *c;                                // [rows, d] attention value
  const float* dc;                         // [rows, d] gradient of the attention value
  float *dK, *dV, *dkt, *dvt, *dq;
  const float* alibi;                      // [H] or NULL
  float scale, scale_log2;
  int B, H, d, N;
};

// Eight consecutive entries of a 64-wide head per lane, eight lanes per (query, key) pair: a dot product costs three shuffles for four pairs.
struct F8 { float v[8]; };
__device__ __forceinline__ F8 ld8(const float* p) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  return F8{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}
__device__ __forceinline__ void st8(float* p, const F8& x) {
  *reinterpret_cast<float4*>(p) = make_float4(x.v[0], x.v[1], x.v[2], x.v[3]);
  *reinterpret_cast<float4*>(p + 4) = make_float4(x.v[4], x.v[5], x.v[6], x.v[7]);
}
__device__ __forceinline__ float dot8(const F8& a, const F8& b) {
  float s = 0.f;
#pragma unroll
  for (int e = 0; e < 8; ++e) s = fmaf(a.v[e], b.v[e], s);
  return s;
}
__device__ __forceinline__ float group_sum(float v) {          // over the eight lanes of a group
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  return v;
}

// qkRMS backward of dk of one (position, sequence, head) and the bf16 operand row [dk_raw | dv] of the next product; a group of eight
// lanes, eight entries each; all lanes of the warp take part, those that are not live store nothing.
__device__ __forceinline__ void pair_operand(const F8& dk, const F8& dv, const F8& u, const __nv_bfloat16* g_k, int h, int t, float eps, int qk, float* dkraw,
                                             __nv_bfloat16* op_k, __nv_bfloat16* op_v, bool live) {
  F8 r = dk;
  if (qk) {
    F8 ty;
#pragma unroll
    for (int e = 0; e < 8; ++e) ty.v[e] = dk.v[e] * gain_at(g_k, h * kHeadDim + 8 * t + e);
    const float ss = group_sum(dot8(u, u)), tu = group_sum(dot8(ty, u));
    const float inv = rsqrtf(ss / kHeadDim + eps), mean = tu * inv / kHeadDim;
#pragma unroll
    for (int e = 0; e < 8; ++e) r.v[e] = inv * (ty.v[e] - u.v[e] * inv * mean);
  }
  if (!live) return;
  st8(dkraw, r);
  unsigned a[4], b[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const __nv_bfloat162 x = __floats2bfloat162_rn(r.v[2 * e], r.v[2 * e + 1]), y = __floats2bfloat162_rn(dv.v[2 * e], dv.v[2 * e + 1]);
    a[e] = *reinterpret_cast<const unsigned*>(&x); b[e] = *reinterpret_cast<const unsigned*>(&y);
  }
  *reinterpret_cast<uint4*>(op_k) = make_uint4(a[0], a[1], a[2], a[3]);
  *reinterpret_cast<uint4*>(op_v) = make_uint4(b[0], b[1], b[2], b[3]);
}
struct WidePair { const float* kraw; float* dkraw; const __nv_bfloat16* g_k; __nv_bfloat16* op; float eps; int qk; };      // op [B][2 d]

}  // namespace rt
