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

// Operand rows of the tensor-core products: one bf16 value per entry, or (terms = 3) three whose sum is the fp32 value to 2^-24, at rows
// term_stride apart.
struct WidePair { const float* kraw; float* dkraw; const __nv_bfloat16* g_k; __nv_bfloat16* op; float eps; int qk, terms; long long term_stride; };      // op [B][2 d]
__device__ __forceinline__ unsigned split_pair(float& a, float& b) {       // bf16 of both, which keep the rest
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  const unsigned w = *reinterpret_cast<const unsigned*>(&v);
  a -= __uint_as_float(w << 16); b -= __uint_as_float(w & 0xffff0000u);
  return w;
}
__device__ __forceinline__ void store_operand8(__nv_bfloat16* at, F8 x, int terms, long long term_stride) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (k >= terms) break;
    unsigned w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) w[e] = split_pair(x.v[2 * e], x.v[2 * e + 1]);
    *reinterpret_cast<uint4*>(at + k * term_stride) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}
__device__ __forceinline__ void store_operand4(__nv_bfloat16* at, float a, float b, float c, float d, int terms, long long term_stride) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (k >= terms) break;
    const unsigned lo = split_pair(a, b), hi = split_pair(c, d);
    *reinterpret_cast<uint2*>(at + k * term_stride) = make_uint2(lo, hi);
  }
}
// qkRMS backward of dk of one (position, sequence, head) and the operand row [dk_raw | dv] of the next product; a group of eight
// lanes, eight entries each; all lanes of the warp take part, those that are not live store nothing.
__device__ __forceinline__ void pair_operand(const F8& dk, const F8& dv, const F8& u, const WidePair& w, int b, int d, int h, int t, float* dkraw, bool live) {
  F8 r = dk;
  if (w.qk) {
    F8 ty;
#pragma unroll
    for (int e = 0; e < 8; ++e) ty.v[e] = dk.v[e] * gain_at(w.g_k, h * kHeadDim + 8 * t + e);
    const float ss = group_sum(dot8(u, u)), tu = group_sum(dot8(ty, u));
    const float inv = rsqrtf(ss / kHeadDim + w.eps), mean = tu * inv / kHeadDim;
#pragma unroll
    for (int e = 0; e < 8; ++e) r.v[e] = inv * (ty.v[e] - u.v[e] * inv * mean);
  }
  if (!live) return;
  st8(dkraw, r);
  __nv_bfloat16* op = w.op + (long long)b * 2 * d + h * kHeadDim + 8 * t;
  store_operand8(op, r, w.terms, w.term_stride);
  store_operand8(op + d, dv, w.terms, w.term_stride);
}

}  // namespace rt
