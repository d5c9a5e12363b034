// Host-side launch interface of the RT kernels (internal; the public ABI is include/rt.h).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "rt_common.cuh"

namespace rt {

// Everything the per-token chain needs.  Position-major buffers are [row, B, d] with
// row = t - row_off (prefill: row_off = 0; decode: the single row 0 stands for position pos).
struct LeafParams {
  int B, d, H, dff;
  int norm_flags;
  float eps, scale_log2, alpha;
  const void *w_o, *w_up, *w_down, *w_k, *w_v;   // storage type
  const void *g_mlp, *g_kv, *g_k;                // storage type or NULL
  const float* alibi;                            // [H] slopes of the ALiBi distances (natural-log units) or NULL
  const void* x;  long long x_bs, x_ts;          // x[b, t, :] = x + b*x_bs + (t-row_off)*x_ts   (elements)
  void* z;        long long z_bs, z_ts;
  void *k_cache, *v_cache;                       // [N_max, B, d] storage type
  const void* q;                                 // [rows, B, d] storage type
  float *st_o, *st_m, *st_l;                     // online-softmax state: o [rows,B,d], m,l [rows,B,H] (m in log2 units)
  int t0, t1;                                    // positions [t0, t1) are processed by this launch
  int row_off;
  // tensor-core leaf kernel on a slice of the batch: the rows of q, the state and the caches are [row][Bs][...] and this
  // launch's sequence b is column b0 + b of them (x and z are passed already offset); Bs = 0 means Bs = B, b0 = 0
  int Bs, b0;
  int attn_begin;                                // first key position the in-launch attention covers (0 = whole prefix)
  float *ex_h, *ex_g, *ex_z, *ex_k;              // exchange vectors [B,d], [B,dff], [B,d], [B,d]
  float* ex_part;                                // partial attention states [B*H, max_chunks, 66]
  int max_chunks;
  int weights_in_smem;                           // 1: each CTA keeps its weight rows in shared memory
  unsigned bar_base;                             // arrivals counted by earlier launches of the same call (bar_count is
                                                 // zeroed once per API call and only ever grows)
  unsigned seq_base;                             // token steps enqueued before this launch in the same call (flag values)
  int timers;                                    // 1: CTA 0 accumulates per-phase times in the sync area (costs a few per cent)
  SyncArea* sync;
};

struct LeafLaunch { int grid, block; size_t smem; int weights_in_smem; };

// Chooses grid / shared memory for the leaf kernel on the current device.
cudaError_t leaf_plan(int dtype, int B, int d, int dff, LeafLaunch* out);
cudaError_t leaf_launch(int dtype, const LeafParams& p, const LeafLaunch& l, cudaStream_t s);
// Barrier arrivals one launch over [t0,t1) adds to bar_count.
inline unsigned leaf_barrier_arrivals(int t0, int t1, int grid) { return (unsigned)(t1 - t0) * 5u * (unsigned)grid; }

// launches a 2-CTA kernel whose barrier cannot complete (tests the bounded-wait path)
cudaError_t wait_expiry_selftest_launch(SyncArea* sync, cudaStream_t s);

// bf16 / tiled-schedule leaf kernel (tensor-core mat-vecs, flag-carrying exchange words).
struct LeafMmaLaunch { int grid, block; size_t smem; int leaf; int q_smem; };
// vectors: c, h, z, g of every position of the launch, packed bf16 [positions][16 (3 d + dff)], filled with ones before; raw k|v as words beside their step number [B,2d]
struct LeafMmaBuffers { unsigned char* vectors; unsigned long long* ll_kv; };
inline size_t leaf_mma_set_bytes(int d, int dff) { return (size_t)32 * (3 * (size_t)d + (size_t)((dff + 31) & ~31)); }
bool leaf_mma_plan(int B, int d, int H, int dff, int want_leaf, LeafMmaLaunch* out);
// the same decision for a device with `sms` multiprocessors and `max_smem` bytes of shared memory per CTA (no CUDA call)
bool leaf_mma_shape(int B, int d, int H, int dff, int want_leaf, int sms, size_t max_smem, LeafMmaLaunch* out);
constexpr int kB200Sms = 148;                    // the part this library is written for: what the pure-host planner assumes
constexpr size_t kB200SmemPerCta = 232448;
cudaError_t leaf_mma_launch(const LeafParams& p, const LeafMmaLaunch& l, const LeafMmaBuffers& buf, cudaStream_t s);

// Leaf kernel for layers that fit one cluster's shared memory (rt_leaf_small.cu).
struct LeafSmallLaunch { int nb, leaf; size_t smem; float step_us; };      // step_us: estimate of the time per position
bool leaf_small_shape(int dtype, int B, int d, int H, int dff, int leaf, size_t max_smem, LeafSmallLaunch* out);
cudaError_t leaf_small_launch(int dtype, const LeafParams& p, const LeafSmallLaunch& l, cudaStream_t s);

// Leaf kernel for several independent (layer, slice) jobs side by side, a group of SMs each (bf16; rt_leaf_group.cu).
constexpr int kGroupJobs = 8;
struct GroupJob {
  const void* packed;                            // W_o, W_up, W_down, W_k, W_v in the order of use (leaf_group_pack)
  const void *g_mlp, *g_kv, *g_k;                // storage type or NULL
  const float* alibi;
  const void* q;                                 // [row, Bs, d]
  const float *st_o, *st_m, *st_l;
  const void* x; long long x_bs, x_ts;           // x[b, t, :] of this job's first sequence
  void* z; long long z_bs, z_ts;
  void *k_cache, *v_cache;                       // [N_max, Bs, d]
  int row_off;                                   // position of row 0 of q and of the state
  int t0, t1;                                    // positions
  int key0;                                      // first position whose pair is not in the states yet (key0 <= t0)
  int B, b0;                                     // sequences of the slice, first column in q / state / caches
  unsigned char* words;                          // exchange area of the job's place, filled with ones once per API call
  unsigned steps;                                // token steps enqueued on that place before this launch in the same call
};
struct GroupCommon {
  int d, H, dff, Bs;                             // Bs: sequences per row of q, state and caches
  int norm_flags;
  float eps, scale_log2, alpha;
  SyncArea* sync;
};
constexpr int kGroupPackLayers = 8;
struct GroupPackLayer { const void *w_o, *w_up, *w_down, *w_k, *w_v; void* out; };
struct GroupPackArgs { int d, dff, g; GroupPackLayer layer[kGroupPackLayers]; };
bool leaf_group_shape(int B, int d, int H, int dff, int places, size_t max_smem);   // B: sequences of one job; groups of 148 / places SMs
float leaf_group_step_us(int B, int d, int dff, int places);                         // estimate of the time per position
size_t leaf_group_words_bytes(int d, int dff);   // exchange area of one place
size_t leaf_group_packed_bytes(int d, int dff, int places);
cudaError_t leaf_group_pack(const GroupPackLayer* layers, int n, int d, int dff, int places, cudaStream_t s);
cudaError_t leaf_group_launch(const GroupCommon& c, const GroupJob* jobs, int n_jobs, int places, cudaStream_t s);   // n_jobs <= places

// Reverse loop of the backward pass over one leaf of at most 64 positions (bf16 weights, at most eight sequences; rt_backward_loop.cu).
// Arrays are position-major fp32 [position, Bs, d | dff] unless said otherwise; dkraw, dvf, dr, dpre, du, dc are filled with 0xFF bytes before.
struct BwdLeafParams {
  int B, b0, Bs, d, H, dff;
  int s0, e0;
  int z_norm, pre, qk;
  float eps, alpha, scale, scale_log2;
  const void *wkT, *wvT, *wdnT, *wupT, *woT;     // transposed weights, bf16
  const void *g_k, *g_kv, *g_mlp;                // bf16 or NULL
  const float* alibi;
  const void* z; long long z_bs, z_ts;           // layer output [B, N, d] bf16
  const float* dz; long long dz_bs, dz_ts;
  const float *q, *k, *v, *kt, *vt, *c, *lse, *kraw, *h, *act;
  float *dK, *dV, *dvf, *dkraw, *dr, *Gz, *dpre, *du, *dh, *dc, *dkt, *dvt, *D;
  SyncArea* sync;
};
int bwd_leaf_slice(int B, int d, int H, int dff, int max_b);
cudaError_t bwd_leaf_launch(const BwdLeafParams& p, cudaStream_t s);

// Pre-pass (Algorithm 1, line 1 and the temporary pair of line 7, hoisted out of the loop).
struct PrepassParams {
  int B, N, d, H;
  int norm_flags;
  float eps, scale_log2;
  const void* x; long long x_bs, x_ts;           // x[b, r, :]
  const void *w_q, *w_k, *w_v, *g_attn, *g_q, *g_k;
  void* n;                                       // [N*B, d] normalised input (scratch)
  void *q, *kt, *vt;                             // [N, B, d]
  float *st_o, *st_m, *st_l;
  int mats;                                      // which projections to compute: bit 0 q, bit 1 k, bit 2 v (0 = all three)
  int no_seed;                                   // 1: leave the running stats alone (projection only)
  int skip_rms;                                  // 1: `n` already holds the normalised rows
  int chained;                                   // 1: launch the projection as a programmatic dependent launch
  SyncArea* sync;
};
cudaError_t prepass_launch(int dtype, const PrepassParams& p, cudaStream_t s);
// The pre-passes of up to kPrepassBatch layers' rows together (same B, d and flags): three launches for all of them.
constexpr int kPrepassBatch = 8;
struct PrepassBatch { PrepassParams p[kPrepassBatch]; };
cudaError_t prepass_batch_launch(int dtype, const PrepassParams* p, int n, cudaStream_t s);
// tensor-core projection (bf16, d a multiple of 128)
bool qkv_gemm_tc_supported(const PrepassParams& p);
cudaError_t qkv_gemm_tc_launch(const PrepassParams& p, SyncArea* sync, cudaStream_t s);
cudaError_t qkv_gemm_tc_batch_launch(const PrepassBatch& b, int n, int rows_max, SyncArea* sync, cudaStream_t s);

// Cross-block tile (Algorithm 2 on a [q0,q1) x [k0,k1) block for every sequence and head).
struct TileParams {
  int B, d, H;
  float scale_log2;
  const float* alibi;                            // [H] slopes of the ALiBi distances (natural-log units) or NULL
  const void* q;                                 // [N, B, d]
  const void *k_cache, *v_cache;                 // [N_max, B, d]
  float *st_o, *st_m, *st_l;
  int q0, q1, k0, k1;
  int batch, batch_stride, q_limit;              // batch > 1: blockIdx.z-th copy of the tile, shifted by z * batch_stride rows
                                                 // (one level of Algorithm 1 in one launch); q_limit > 0 clips the queries
  int causal;                                    // 1: only pairs with key position < query position
  int causal_full;                               // with causal (tensor-core kernel): a CTA's key blocks end at its own query tile, so one
                                                 // launch over [q0,q1) x [k0,k1) covers every query's whole causal prefix; heavy tiles first
  int chained;                                   // row_attn only: launch as a programmatic dependent launch
  void* c_out;                                   // row_attn only: also write the attention value o/l of the row, [B, d] storage type
  int q_pos0;                                    // position of query row 0 (ALiBi distances; kernels without a mask only)
  int rows_q, rows_kv;                           // rows held by the query buffer / the caches (tensor-map bounds)
  SyncArea* sync;
};
cudaError_t tile_launch(int dtype, const TileParams& p, cudaStream_t s);
// tensor-core version (bf16, key count a multiple of 64)
cudaError_t tile_tc_launch(const TileParams& p, int rows_q, int rows_kv, SyncArea* sync, cudaStream_t s);
// one tile of each of n layers (n <= kGroupJobs, key counts multiples of 64, the same B, d, H; slopes in all or none)
cudaError_t tile_tc_batch_launch(const TileParams* p, int n, SyncArea* sync, cudaStream_t s);
cudaError_t tile_simt_launch(int dtype, const TileParams& p, cudaStream_t s);
// bf16 tiles of n layers (1 <= n <= kGroupJobs, the same B, d, H; pairs by whole blocks of 32), probabilities in fp32
cudaError_t tile_rows_batch_launch(const TileParams* p, int n, cudaStream_t s);
// one query row (position q0) per (sequence, head) against the pairs [k0, k1): the in-leaf step of wide batches
cudaError_t row_attn_launch(int dtype, const TileParams& p, cudaStream_t s);

// Decode step of up to kDecMaxLayers layers in one cooperative launch (bf16, at most 16 sequences; rt_decode.cu).
constexpr int kDecMaxLayers = 16;
struct DecLayer {
  const void *w_q, *w_k, *w_v, *w_o, *w_up, *w_down;
  const void *g_attn, *g_mlp, *g_kv, *g_q, *g_k;   // storage type or NULL (g_kv: g_attn where the layer has none)
  const float* alibi;
  void *k_cache, *v_cache;
};
struct DecodeParams {
  int n_layers, B, d, H, dff;                      // B: sequences of this launch
  int full;                                        // 1: the vectors between the phases stay fp32 (at most eight sequences)
  int pos;                                         // positions in the caches
  int Bs, b0;                                      // sequences per cache row, first of this launch
  int norm_flags;
  float eps, scale_log2, alpha;
  const void* x; long long x_bs;                   // input rows [B, d] (row stride x_bs), or NULL:
  const void* emb; const int32_t* ids; int vocab;  // rows of the embedding
  void* z_out; long long z_bs;                     // the last layer's output rows
  const void* next_bytes; size_t next_size;        // what the following kernel reads (L2 prefetch); may be NULL
  unsigned char* words; size_t words_size;         // exchange area, decode_words_bytes(...)
  SyncArea* sync;
  DecLayer layer[kDecMaxLayers];
  int quads, chunks, chunk_len, warps_per_cta, pf_keys;   // attention split, set by the launcher
};
bool decode_shape(int B, int d, int H, int dff);   // whether the kernel takes the slices of a batch of B
// Sequences per launch: a batch above 16 (full: above eight) runs as slices of equal size (the sequences are independent), the last one with what is left.
int decode_slice(int B, bool full);
// Bytes of exchange area for the slices of a batch of at most B, one after the other (0: the kernel does not take the shape).
size_t decode_words_bytes(int n_layers, int B, int d, int H, int dff);
cudaError_t decode_launch(const DecodeParams& p, cudaStream_t s);

// Stack helpers.
cudaError_t embed_launch(int dtype, const void* emb, const int32_t* ids, int B, int N, int d, int vocab,
                         void* x, cudaStream_t s);
cudaError_t head_launch(int dtype, const void* emb, const void* g_final, const void* hidden, long long h_bs,
                        int B, int d, int vocab, int norm_flags, float eps, float* logits, cudaStream_t s);

// Token loop of wide batches in one cooperative launch per leaf (bf16; rt_wide_loop.cu).
constexpr int kWideGroupsMax = 8;                // groups of at most 128 sequences
// fills of the operand ring over the whole contraction, tile width, tiles, parts of the contraction, fills the ring holds
struct WideStage { int fills, bn, tiles, splits, slots; };
struct WideFwdParams {
  int B, d, H, dff, norm_flags;
  float eps, scale_log2, alpha;
  const void *w_o, *w_up, *w_down, *w_k, *w_v, *g_mlp, *g_kv, *g_k;
  const float* alibi;
  const void* x; long long x_bs, x_ts;
  void* z; long long z_bs, z_ts;
  const void* q;                                 // [N, B, d]
  const float *st_o, *st_m, *st_l;               // state of every row before its leaf
  void *k_cache, *v_cache;                       // [N_max, B, d]
  int t0, t1;                                    // positions of the leaf
  unsigned steps;                                // positions since the counters were zeroed
  unsigned* counters;                            // wide_counter_bytes(B)
  float *h, *partial, *ssq_h, *ssq_z;            // [B, d], [8, B, d], [wide_ssq_floats, B] (ssq_z is set by the launcher)
  void *c16, *u16, *g16, *r16;                   // bf16 operand rows [B, d], [B, d_ff] (g16)
  SyncArea* sync;
  int R, G, a_bytes;                             // set by the launcher: sequences and SMs per group, bytes of an operand block
  WideStage st[4];                               // W_o, W_up, W_down, W_k | W_v
};
struct AttnBufs;
struct WidePair;
constexpr int kWideTermRows = 32;                // rows between the terms of a three-term operand (batches of at most 32)
struct WideBwdParams {
  int B, terms, d, H, dff, z_norm, pre;
  float eps, alpha;
  const void *wkvT, *wdnT, *wupT, *woT;          // bf16 [d, 2 d], [d_ff, d], [d, d_ff], [d, d]
  const void *g_kv, *g_mlp;
  const void* z; long long z_bs, z_ts;
  const float* dz; long long dz_bs, dz_ts;
  const float *h, *act;                          // fp32 position-major [N, B, ...], as the arrays below
  float *dr, *Gz, *dpre, *du, *dh, *dc;
  float* partial;                                // [8, B, d]
  void *s16, *p16;                               // bf16 operand rows [B, d], [B, d_ff]
  int s0, e0;                                    // positions of the leaf, last one first
  unsigned steps;                                // positions since the counters were zeroed
  unsigned* counters;
  SyncArea* sync;
  int R, G, a_bytes;                             // set by the launcher
  WideStage st[4];                               // W_k | W_v, W_down, W_up, W_o
};
int wide_backward_groups(int B, int d, int dff); // 0: not taken
cudaError_t wide_backward_launch(WideBwdParams p, const AttnBufs& a, const WidePair& wp, cudaStream_t s);
int wide_loop_groups(int B, int d, int dff);     // 0: not taken
size_t wide_counter_bytes(int B);
int wide_ssq_floats(int d);
cudaError_t wide_forward_launch(WideFwdParams p, cudaStream_t s);

// Position-wise part of the parallel sweep (Sec. 6, activation checkpointing): dense products over all rows.
enum { DENSE_RES_X = 0, DENSE_GELU = 1, DENSE_RES_H = 2, DENSE_F32 = 3, DENSE_GELU_BWD = 4 };
struct DenseParams {
  int M, N, K, B;                                // C[M,N] = A[M,K] W[N,K]^T; rows m = position * B + sequence
  const void *A, *W;                             // storage type, K contiguous
  int epi;                                       // DENSE_RES_X: h = x + alpha C (fp32);  DENSE_GELU: out = GELU(C);
                                                 // DENSE_RES_H: out = h + alpha C (storage type, caller's strides)
                                                 // DENSE_F32: h = alpha C, or h += alpha C with `accumulate` (fp32 [M, N])
                                                 // DENSE_GELU_BWD: h = C GELU'(x) (x, h fp32 [M, N]), out = h in the storage type (tensor cores, not split)
  float alpha;
  int accumulate;                                // DENSE_F32 only
  const void* x; long long x_bs, x_ts;           // x[b, r, :] (DENSE_RES_X)
  float* h;                                      // [M, N] fp32 (written by DENSE_RES_X, read by DENSE_RES_H)
  void* out; long long o_bs, o_ts;               // DENSE_GELU: [M, N];  DENSE_RES_H: out[b, r, :]
  float* partial; size_t partial_bytes;          // optional scratch for a split contraction (few rows): [splits, M, N] fp32
  int splits;                                    // set by the launcher
  int keep_partial;                              // 1: leave the partial sums in `partial` ([splits, M, N], one split included) and reduce nothing;
                                                 // the number of splits comes back through dense_launch's last argument
  int chained;                                   // 1: launch the product (and its reduction) as programmatic dependent launches
  // optional: also write RMS_g(row) of the epilogue's result (h or z) for the next product.  Only a split
  // contraction does this (its reduction kernel owns whole rows); `normed` tells the caller whether it happened.
  void* norm_out; const void* norm_gain; float norm_eps; int norm_pre;
  // DENSE_QKV (persistent CTA pairs only): three products A W_q^T, A W_k^T, A W_v^T in one launch, N = d columns each;
  // qkRMS over each head's 64 columns of q and k (qk_norm), bf16 outputs [M, d]
  const void *W2, *W3;                           // W = W_q, W2 = W_k, W3 = W_v
  void *q_out, *k_out, *v_out;
  const void *g_q, *g_k;
  int qk_norm; float qk_eps;
};
constexpr int DENSE_QKV = 100;
// The q / k~ / v~ projections of the pre-pass as one launch of persistent CTA pairs (bf16, d a multiple of 256, at least a
// wave of tiles); false when the shape does not qualify (the caller then takes qkv_gemm_tc_launch's own kernel).
bool dense_qkv_pair_supported(int M, int d);
cudaError_t dense_qkv_pair_launch(const DenseParams& p, SyncArea* sync, cudaStream_t s);
cudaError_t dense_launch(int dtype, const DenseParams& p, SyncArea* sync, cudaStream_t s, bool* normed = nullptr, int* splits = nullptr);
cudaError_t attn_value_launch(int dtype, const float* st_o, const float* st_l, void* c, long long rows, int d, int H, cudaStream_t s,
                              bool chained = false);
cudaError_t rms_rows_f32_launch(int dtype, const float* h, const void* g, void* u, int rows, int d, float eps, int pre, cudaStream_t s,
                                bool chained = false);

// Event-pair span for rt_profile_enable / rt_profile_read from other translation units (classes: 0 sweeps / pre-pass,
// 1 per-position steps, 2 attention tiles, 3 everything else).  Does nothing while profiling is off.
struct ProfSpanScope {
  void* impl = nullptr;
  ProfSpanScope(cudaStream_t s, int cls);
  ~ProfSpanScope();
  ProfSpanScope(const ProfSpanScope&) = delete;
  ProfSpanScope& operator=(const ProfSpanScope&) = delete;
};

}  // namespace rt
