// C ABI of the library (see include/rt.h): argument checks, workspace layout, and the
// schedule of Algorithm 1 at leaf granularity -- solve a leaf, then let the next query block
// attend to the block of pairs that just became complete.
#include <math.h>
#include <string.h>

#include <mutex>
#include <vector>

#include "rt_kernels.h"
#include "rt_wave.h"

using namespace rt;

namespace {

constexpr int kMaxChunks = 32;
constexpr int kSmallBatchMax = 64;      // above this the per-token chain runs as dense products (tiled prefill only)
constexpr int kAutoLeaf = 64;

struct WsLayout {
  size_t sync, q, kt, vt, n, st_o, st_m, st_l, ex_h, ex_g, ex_z, ex_k, ex_part, ll, ll_bytes, form, form_bytes, sets, dec_words, dec_words_bytes, hid0, hid1,
      blk_h, blk_u, blk_c, blk_g, total;
};

size_t esize_of(int dtype) { return dtype == RT_BF16 ? 2 : 4; }

bool config_ok(const rt_config* c) {
  if (!c) return false;
  if (c->d_model <= 0 || c->n_heads <= 0 || c->head_dim <= 0 || c->d_ff <= 0) return false;
  if ((long long)c->n_heads * c->head_dim != c->d_model) return false;
  if (c->dtype != RT_F32 && c->dtype != RT_BF16) return false;
  if (c->sched != RT_SCHED_TILED && c->sched != RT_SCHED_NAIVE) return false;
  if (c->leaf != 0 && (c->leaf < 16 || c->leaf > 256 || (c->leaf & (c->leaf - 1)))) return false;
  if (!(c->rms_eps >= 0.f) || !isfinite(c->softmax_scale) || !isfinite(c->residual_scale)) return false;
  if (c->norm_flags & ~(RT_NORM_PRE | RT_NORM_QK | RT_NORM_SKIP_Z)) return false;
  if (c->recur_block < 0) return false;
  if (c->flags & ~RT_FLAG_BACKWARD_STEP_LAUNCHES) return false;
  return true;
}

rt_status config_supported(const rt_config* c, int B, bool wide_ok = false) {
  if (c->head_dim != kHeadDim) return RT_ERR_UNSUPPORTED;
  if (c->d_ff % 4) return RT_ERR_UNSUPPORTED;
  if (B > kSmallBatchMax && !(wide_ok && c->sched == RT_SCHED_TILED)) return RT_ERR_UNSUPPORTED;
  return RT_OK;
}

int leaf_size(const rt_config* c) { return c->leaf ? c->leaf : kAutoLeaf; }

// Which form of the per-token chain a prefill with this configuration and batch runs, and the granularity of
// Algorithm 1's tiles that goes with it.  Used by run_layer and by rt_plan_counters, so that the modelled schedule is
// the one that runs (the tensor-core leaf kernel's leaf depends on the shared memory of the part; the planner assumes
// a B200).
enum ChainPath { kPathGeneric = 0, kPathMma = 1, kPathWide = 2, kPathBlocks = 3, kPathMmaSplit = 4, kPathGroups = 5 };
struct Schedule { ChainPath path; int leaf; int sub; };      // sub: sequences per slice (kPathMmaSplit, kPathGroups)
constexpr int kWideLeafDefault = 16;    // leaf of the dense-product token steps.  As launches per position, whose in-leaf attention re-reads the leaf's pairs
                                        // for every position, short leaves win (p512: 16 -> 41.6 ms, 32 -> 42.3, 64 -> 45.9 per layer); in one launch per leaf
                                        // 32 or 64 would be 1.5 to 6 % faster, but the modelled schedule of wide batches is that of 16
constexpr int kWideFrom = 24;            // smallest bf16 batch that runs as dense products rather than through the generic kernel
constexpr int kMmaSplitMax = 48;         // largest batch that runs as slices of at most 16 sequences through the tensor-core leaf kernel
constexpr int kGroupsMax = 64;           // largest batch that runs as slices of at most 16 sequences side by side on groups of SMs
Schedule effective_schedule(const rt_config* c, int B, int N) {
  if (c->recur_block > 1) return {kPathBlocks, c->recur_block, 0};
  if (c->sched == RT_SCHED_TILED) {
    LeafMmaLaunch ml;
    // (a single position does not pay for packing the weights: d = 1024, B = 32 takes 65 us without, 120 us through the generic kernel)
    if (c->dtype == RT_BF16 && B > 16 && B <= kGroupsMax && N > 1) {
      // slices side by side, a group of SMs each (rt_leaf_group.cu), unless the layer would otherwise take the generic kernel: that one holds
      // the vectors between the phases in fp32, the others round them to bf16 (d = 512, B = 20, leaves of 128: error of k against 64 bits
      // 1.9e-3 and 3.0e-3)
      const int n_sub = ceil_div(B, 16), sub = ceil_div(B, n_sub);
      if (leaf_group_shape(sub, c->d_model, c->n_heads, c->d_ff, n_sub, kB200SmemPerCta) &&
          (B >= kWideFrom || leaf_mma_shape(sub, c->d_model, c->n_heads, c->d_ff, c->leaf, kB200Sms, kB200SmemPerCta, &ml)))
        return {kPathGroups, c->leaf ? c->leaf : kAutoLeaf, sub};
    }
    if (c->dtype == RT_BF16 && B > 16 && B <= kMmaSplitMax) {
      // What the group kernel does not take (a single position, layers that fit no group): sequences are independent (Sec. 2.2 states
      // the layer per sequence) and a token step of the tensor-core leaf kernel costs 9 - 14 us whatever its batch, against 53 us for the
      // dense-product step at B = 32: up to 48 sequences run as 2 or 3 slices of at most 16 through that kernel, leaf by leaf, and share the cross tiles.
      const int n_sub = (B + 15) / 16, sub = (B + n_sub - 1) / n_sub;
      if (leaf_mma_shape(sub, c->d_model, c->n_heads, c->d_ff, c->leaf, kB200Sms, kB200SmemPerCta, &ml))
        return {kPathMmaSplit, ml.leaf, sub};
    }
    // bf16 batches beyond that (or whose slices the tensor-core leaf kernel does not take) run as dense products from
    // 24 sequences on, where they overtake the generic kernel (measured at d = 1024: 53 us per token step at B = 32
    // against 99 us); fp32 keeps the generic kernel up to its limit
    if (B > kSmallBatchMax || (c->dtype == RT_BF16 && B >= kWideFrom)) return {kPathWide, c->leaf ? c->leaf : kWideLeafDefault, 0};
    if (c->dtype == RT_BF16 && leaf_mma_shape(B, c->d_model, c->n_heads, c->d_ff, c->leaf, kB200Sms, kB200SmemPerCta, &ml))
      return {kPathMma, ml.leaf, B};
  }
  return {kPathGeneric, leaf_size(c), 0};
}

// The layers of a stack side by side (rt_leaf_group.cu): layer l works on a leaf that layer l-1 finished in an earlier
// launch, up to `places` layers in a launch, a group of SMs each.  places = 0: one layer after the other.
struct Wave { int places, leaf, packs, exact; };      // packs: layers whose packed weights are held at a time; deeper stacks run band after band.  exact: see wave_exact_tile
// longest leaf of layers side by side (what the workspace holds rows for)
int wave_leaf_max(const rt_config* c, int N) { return c->leaf ? c->leaf : N <= 128 ? 16 : N <= 1024 ? 32 : 64; }
constexpr int kWaveBlock = 64;           // earlier pairs come by whole blocks of this many from the tile kernel, the rest of them inside the leaf kernel
// Stacks of up to kWaveExactN positions whose layers run, or by the four-place line of stack_wave could run, side by side: the whole blocks of 64 pairs before a
// leaf that begins at t0 < kWaveExactMax come from a tile kernel with fp32 probabilities, not from the tensor-core one, which rounds them to bf16.  All other
// stacks give the bits of the same layers one by one, whose tiles begin with the second block.
constexpr int kWaveExactN = 1024, kWaveExactMax = 192;
bool wave_exact_tile(bool exact, int t0) { return exact && t0 < kWaveExactMax; }
// Estimates (us) of a stack's token loops, side by side and one after the other.  Fitted to 16 widths from d = 64 to 1024, 1 to 16 sequences, 2 to 8 places and leaves of
// 16, 32 and 64 (256 positions; 5 % off on average from d = 320 on) and checked on long stacks, ms measured / estimated, side by side and one after the other: 8 layers of d = 1024,
// B = 1, N = 2048 82.6 / 75, 139 / 145, 16384 743 / 651, 1116 / 1161, 65536 3651 / 3519, 4480 / 4704; B = 16, N = 2048 111 / 101, 190 / 192, 16384 1146 / 1040, 1601 / 1606, 65536
// 7596 / 7570, 7472 / 7391; d = 512, B = 16, N = 32768 1149 / 1175, 2785 / 2853; 2 layers of d = 1024, B = 16, N = 16384 372 / 402, 401 / 402, 32768 861 / 947, 845 / 843.
// Tiles are what grows with the length: a leaf reads its layer's whole cache so far, so side by side they cost (N / 64)^2 / 2 blocks of 64 pairs x 64 queries a layer and (sequence,
// head), 1.15 us each behind one another or 4.2 ns where they fill the chip; the same pairs cost 1.2 ns in Algorithm 1's larger tiles.  So one after the other, whose
// cache traffic is N log N, is the faster form again from some length on: some 65 thousand positions for 8 layers of d = 1024, B = 16, some 20 thousand for 2.
// Widths that are no multiple of 128 take the fp32 pre-pass, whose time per launch of leaves is 0.06 d us a layer and more.
int band_begin(int n_layers, int bands, int b) { return (int)((long long)n_layers * b / bands); }      // (bands of about the same depth)
bool tensor_prepass(const rt_config* c) { return c->d_model % 128 == 0; }
float wave_us(const rt_config* c, int B, int N, int n_layers, const Wave& w) {
  const int places = w.places, leaf = w.leaf, bands = ceil_div(n_layers, w.packs);
  const float d = (float)c->d_model, tiles = (float)(places * B * c->n_heads), blocks = (float)N / (float)kWaveBlock;
  long long launches = 0;
  for (int b = 0; b < bands; ++b) launches += wave_launches(band_begin(n_layers, bands, b + 1) - band_begin(n_layers, bands, b), ceil_div(N, leaf), places);
  float us = (float)leaf * leaf_group_step_us(B, c->d_model, c->d_ff, places) + 21.0f + 3.5e-4f * (float)(places * B) * d;
  if (!tensor_prepass(c)) us += (float)places * d * (0.06f + 1.2e-6f * (float)B * d);
  // of the whole blocks that come before a leaf, on average half: a launch for each power of two that their number consists of
  if (blocks > 1.0f) us += (1.0f - 1.0f / blocks) * ((0.5f * log2f(blocks) + 0.9f) * (9.0f + 0.01f * tiles) + 0.5f * blocks * fmaxf(1.15f, 4.2e-3f * tiles));
  return (float)launches * us;
}
float alone_us(const rt_config* c, int B, int N, int n_layers) {
  const float d = (float)c->d_model, blocks = (float)N / (float)kWaveBlock;
  const float step = 7.4f + 1.3e-3f * d + 8.6e-5f * (float)B * d + (B > 8 ? 1.5f : 0.0f) + (tensor_prepass(c) ? 0.0f : 2.0e-7f * (float)B * d * d);
  return (float)n_layers * ((float)N * step + 0.6e-3f * (float)(B * c->n_heads) * blocks * blocks);
}
struct WaveRows { size_t n, q, kt, vt, st_o, st_m, st_l, total; };
WaveRows wave_rows_layout(const rt_config* c, int B, int leaf) {
  WaveRows W;
  const size_t e = esize_of(c->dtype), d = c->d_model, H = c->n_heads, rows = (size_t)B * leaf;
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o += align_up(bytes, 256); return at; };
  W.n = take(rows * d * e); W.q = take(rows * d * e); W.kt = take(rows * d * e); W.vt = take(rows * d * e);
  W.st_o = take(rows * d * 4); W.st_m = take(rows * H * 4); W.st_l = take(rows * H * 4);
  W.total = o;
  return W;
}

// Groups of SMs working side by side (slices of a batch, or layers of a stack): an exchange area and a packed layer per group, and for a
// stack a leaf's rows of n, q, k~, v~ and the state per group.
struct GroupArea { size_t packed, packed_stride, rows, rows_stride, total; };
GroupArea group_area(const rt_config* c, int places, int packs, int wave_B, int wave_leaf) {
  GroupArea A;
  A.packed = align_up((size_t)places * leaf_group_words_bytes(c->d_model, c->d_ff), 256);
  A.packed_stride = leaf_group_packed_bytes(c->d_model, c->d_ff, places);
  A.rows = A.packed + align_up(A.packed_stride * packs, 256);
  A.rows_stride = wave_leaf ? wave_rows_layout(c, wave_B, wave_leaf).total : 0;
  A.total = A.rows + A.rows_stride * (wave_leaf ? places : 0);
  return A;
}

// `form`: bytes of the area that the groups work in.
Wave stack_wave(const rt_config* c, int B, int N, int n_layers, size_t form) {
  const Wave none = {0, 0, 0, 0};
  if (n_layers < 2 || N < 2 || c->dtype != RT_BF16 || c->sched != RT_SCHED_TILED || c->recur_block > 1) return none;
  LeafMmaLaunch ml;                                            // (a stack of layers for the generic kernel keeps its fp32 vectors)
  if (!leaf_mma_shape(B, c->d_model, c->n_heads, c->d_ff, c->leaf, kB200Sms, kB200SmemPerCta, &ml)) return none;
  // A leaf meets all earlier pairs at once when its queries exist (they depend on the layer below, so Algorithm 1's tiles cannot
  // run ahead): each leaf reads the layer's whole cache so far, in the parts in which those tiles would have brought it.  The group kernel's sums have the order
  // of the leaf kernel, so a stack gives the bits of the same layers called one by one, where those take leaves of kWaveBlock positions;
  // elsewhere long sequences go layer by layer for the sake of these bits.
  if (N > kWaveExactN && ml.leaf != kWaveBlock) return none;
  // How many layers at a time, and by which leaves: the least time estimated.  More places fill and drain the pipeline of layers in fewer launches, but a
  // group of fewer SMs streams and multiplies more weights per SM; short leaves fill it sooner, long ones have fewer launches.
  Wave best = none;
  float least = 0.0f;
  for (int pl = 2; pl <= kGroupJobs && pl <= n_layers; ++pl) {
    if (!leaf_group_shape(B, c->d_model, c->n_heads, c->d_ff, pl, kB200SmemPerCta)) continue;
    for (int lf = c->leaf ? c->leaf : 16; lf <= wave_leaf_max(c, N); lf *= 2) {
      Wave w = {pl, lf, n_layers < kWaveBand ? n_layers : kWaveBand, N <= kWaveExactN};
      while (w.packs > 1 && group_area(c, pl, w.packs, B, lf).total > form) --w.packs;
      if (w.packs < 2) continue;
      const float us = wave_us(c, B, N, n_layers, w);
      if (!best.places || us < least) { best = w; least = us; }
    }
  }
  // Four layers side by side, each in the place of the one four before it, pay where enough of them are at work at the same time: on average n_layers * N /
  // (launches * leaf) of them, 1.3 to 2.3, more the more weights the groups stream (places x MB per layer) and above four sequences.
  const float layer_mb = (3.0f * c->d_model + 2.0f * c->d_ff) * c->d_model * 2e-6f, mma_us = B > 8 ? 10.5f : 8.3f;
  auto four_pay = [&](float step_us) {                         // step_us: the time per position that the layers take alone, at most mma_us
    const int four = n_layers < 4 ? n_layers : 4, lf = c->leaf ? c->leaf : N <= 128 ? 16 : 32, n = ceil_div(N, lf), turn = n > four ? n : four;
    const float at_work = (float)n_layers * (float)N / (float)(((n_layers - 1) / four * turn + (n_layers - 1) % four + n) * lf);
    const float even = (1.26f + 0.008f * (float)four * layer_mb + (B > 4 ? 0.15f : 0.0f)) * (step_us < mma_us ? mma_us / step_us : 1.0f);
    return leaf_group_shape(B, c->d_model, c->n_heads, c->d_ff, four, kB200SmemPerCta) && at_work > even;
  };
  LeafSmallLaunch sl;
  if (leaf_small_shape(c->dtype, B, c->d_model, c->n_heads, c->d_ff, ml.leaf, kB200SmemPerCta, &sl)) {
    // Layers that fit a cluster (rt_leaf_small.cu) hold the values between the phases in fp32 there, in bf16 here (8 layers of d = 128, B = 1, N = 200: error
    // of the last k against 64 bits 4.95e-3 and 5.2e-3; 2 layers of d = 384 2.97e-3 and 3.3e-3).  So more than four places are no reason to take them
    // off it: they go side by side only where four pay against that kernel, which is faster than the tensor-core leaf kernel (taken as mma_us a position).
    if (N > kWaveExactN) return none;                           // (the bits of that kernel)
    if (!four_pay(sl.step_us)) return none;
    if (best.places) return best;
    return {0, 0, 0, N > kWaveBlock};
  }
  // All others go side by side where that is estimated to be faster.  Over 2 to 8 layers of eight widths from d = 448 to 1024, 1, 5 and 16 sequences and 32 to
  // 700 positions (720 stacks, both ways timed) the choice is on average 0.2 % and at most 8 % slower than the better one; with one break-even for all widths
  // stacks of d = 960 went side by side at up to 1.45 times the time (2 layers, N = 129: 2.30 and 3.34 ms; d = 448, N = 100: 1.65 and 1.95) and 4
  // layers of d = 1024, B = 16, N = 64 did not at 1.19 times (2.99 and 2.52).  The line for four places tells which stacks keep fp32 probabilities one after the other.
  if (best.places && 0.95f * least < alone_us(c, B, N, n_layers)) return best;
  return {0, 0, 0, N > kWaveBlock && N <= kWaveExactN && four_pay(mma_us)};
}
// Positions that the tensor-core leaf kernel has arrays of c, h, z and g for: a leaf, or all layers of a prompt shorter than that (one fill serves
// them: 8 layers of one position, d = 1024, 305 -> 291 us).
int set_positions(const rt_config* c, int N, int n_layers) {
  LeafMmaLaunch ml;
  if (!leaf_mma_shape(1, c->d_model, c->n_heads, c->d_ff, c->leaf, kB200Sms, kB200SmemPerCta, &ml)) return 0;
  return (long long)N * n_layers < ml.leaf ? N * n_layers : ml.leaf;
}

// Bytes of the area that the form of the token loop has to itself: the most that any call of at most B sequences, N positions and n_layers
// layers asks for, whichever form it takes, so that a workspace reserved for the longest prompt and the fullest batch serves all the others.
// (What one form asks for by itself does not grow with the shape: from 17 sequences on there are no arrays of the leaf kernel.)
size_t form_bytes(const rt_config* c, int B, int N, int n_layers) {
  if (c->dtype != RT_BF16) return 0;
  if (c->sched != RT_SCHED_TILED || c->recur_block > 1) return 0;
  const int d = c->d_model, H = c->n_heads, f = c->d_ff, B16 = B < 16 ? B : 16;
  size_t most = 0;
  auto need = [&](size_t bytes) { if (bytes > most) most = bytes; };
  need((size_t)set_positions(c, N, n_layers) * leaf_mma_set_bytes(d, f));
  if (N < 2) return most;
  for (int places = 2; places <= kGroupJobs; ++places) {
    if (!leaf_group_shape(1, d, H, f, places, kB200SmemPerCta)) continue;
    if (B > 16 * (places - 1)) need(group_area(c, places, 1, 0, 0).total);
    if (n_layers >= places) need(group_area(c, places, n_layers < kWaveBand ? n_layers : kWaveBand, B16, wave_leaf_max(c, N)).total);
  }
  return most;
}

// more_form: bytes that the area of the token loop's form gets beyond what it needs.
WsLayout ws_layout(const rt_config* c, int B, int N, int n_layers, size_t more_form = 0) {
  WsLayout L;
  const size_t e = esize_of(c->dtype), d = c->d_model, H = c->n_heads, f = c->d_ff;
  const size_t tok = (size_t)B * N;
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o += align_up(bytes, 256); return at; };
  L.sync = take(sizeof(SyncArea));
  L.q = take(tok * d * e);
  L.kt = take(tok * d * e);
  L.vt = take(tok * d * e);
  L.n = take(tok * d * e);
  L.st_o = take(tok * d * 4);
  L.st_m = take(tok * H * 4);
  L.st_l = take(tok * H * 4);
  L.ex_h = take((size_t)B * d * 4);
  L.ex_g = take((size_t)B * f * 4);
  L.ex_z = take((size_t)B * d * 4);
  L.ex_k = take((size_t)B * d * 4);
  L.ex_part = take((size_t)B * H * kMaxChunks * 68 * 4);
  // exchange buffer of the tensor-core leaf kernel: raw k|v as fp32 words beside their step number (c, h, z and g, packed bf16 in fragment order for 16
  // sequence slots, have arrays per position of a leaf, in `form`)
  L.ll_bytes = (size_t)B * 2 * d * 8;
  L.ll = take(L.ll_bytes);
  L.sets = c->dtype == RT_BF16 ? set_positions(c, N, n_layers) : 0;
  L.form_bytes = form_bytes(c, B, N, n_layers) + more_form;
  L.form = take(L.form_bytes);
  // a decode step uses none of the above but the status block: its exchange area begins right behind that
  L.dec_words = L.q;
  const size_t dec = c->dtype == RT_BF16 ? decode_words_bytes(n_layers, B, (int)d, (int)H, (int)f) : 0;
  if (o < L.dec_words + dec) o = L.dec_words + align_up(dec, 256);
  L.dec_words_bytes = o - L.dec_words;
  L.hid0 = take(tok * d * e);
  L.hid1 = take(tok * d * e);
  // recurrence over blocks: the position-wise chain of one block (rows = block length x B)
  L.blk_h = L.blk_u = L.blk_c = L.blk_g = 0;
  if (c->recur_block > 1) {
    const size_t rows = (size_t)B * (c->recur_block < N ? c->recur_block : N);
    L.blk_h = take(rows * d * 4);
    L.blk_u = take(rows * d * e);
    L.blk_c = take(rows * d * e);
    L.blk_g = take(rows * f * e);
  }
  L.total = o;
  return L;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
bool overlaps(const void* a, size_t na, const void* b, size_t nb) {
  const uintptr_t pa = reinterpret_cast<uintptr_t>(a), pb = reinterpret_cast<uintptr_t>(b);
  return pa < pb + nb && pb < pa + na;
}

bool weights_ok(const rt_layer_weights* w) {
  if (!w) return false;
  const void* req[] = {w->w_q, w->w_k, w->w_v, w->w_o, w->w_up, w->w_down};
  for (const void* p : req) if (!p || !aligned16(p)) return false;
  const void* opt[] = {w->g_attn, w->g_mlp, w->g_kv, w->g_q, w->g_k};
  for (const void* p : opt) if (p && !aligned16(p)) return false;
  return true;
}

// ---- optional per-kernel-class timing (rt_profile_enable / rt_profile_read) -----------------
enum ProfClass { kProfPrepass = 0, kProfLeaf = 1, kProfTile = 2, kProfOther = 3, kProfClasses = 4 };
struct ProfSpan { cudaEvent_t a, b; int cls; };
std::mutex g_prof_mu;
bool g_prof_on = false;
bool g_prof_timers = false;      // rt_profile_enable(2): also the in-kernel phase timers of the leaf kernels
std::vector<ProfSpan> g_prof_spans;
constexpr size_t kProfMaxSpans = 1u << 20;

// Records an event pair around the launches issued inside its scope when profiling is on.
struct ProfScope {
  cudaStream_t s; int cls; cudaEvent_t a = nullptr, b = nullptr; bool on = false;
  ProfScope(cudaStream_t s_, int cls_) : s(s_), cls(cls_) {
    std::lock_guard<std::mutex> g(g_prof_mu);
    if (!g_prof_on || g_prof_spans.size() >= kProfMaxSpans) return;
    if (cudaEventCreate(&a) != cudaSuccess) return;
    if (cudaEventCreate(&b) != cudaSuccess) { cudaEventDestroy(a); return; }
    on = cudaEventRecord(a, s) == cudaSuccess;
  }
  ~ProfScope() {
    if (!a) return;
    if (on && cudaEventRecord(b, s) == cudaSuccess) {
      std::lock_guard<std::mutex> g(g_prof_mu);
      g_prof_spans.push_back({a, b, cls});
    } else { cudaEventDestroy(a); cudaEventDestroy(b); }
  }
};

// State of one API call: the stream and the barrier arrivals enqueued so far.
struct CallCtx { cudaStream_t s; unsigned bar_base = 0; unsigned seq_base = 0; unsigned group_steps[kGroupJobs] = {}; bool groups_cleared = false; int sets_left = 0; bool exact = false; };      // sets_left: arrays of c, h, z, g still filled; exact: first tiles with fp32 probabilities

// The exchange areas of the group kernel start from ones (no word written), once per API call.
bool clear_groups(const rt_config* c, int places, unsigned char* ws, const WsLayout& L, CallCtx& ctx) {
  if (ctx.groups_cleared) return true;
  ctx.groups_cleared = true;
  return cudaMemsetAsync(ws + L.form, 0xFF, (size_t)places * leaf_group_words_bytes(c->d_model, c->d_ff), ctx.s) == cudaSuccess;
}
GroupCommon group_common(const rt_config* c, int B, unsigned char* ws, const WsLayout& L) {
  GroupCommon g;
  memset(&g, 0, sizeof(g));
  g.d = c->d_model; g.H = c->n_heads; g.dff = c->d_ff; g.Bs = B; g.norm_flags = c->norm_flags; g.eps = c->rms_eps;
  g.scale_log2 = c->softmax_scale * kLog2e; g.alpha = c->residual_scale; g.sync = (SyncArea*)(ws + L.sync);
  return g;
}

// One layer on position-major scratch; x / z given with explicit strides.
rt_status run_layer(const rt_config* c, const rt_layer_weights* w, const void* x, long long x_bs, long long x_ts,
                    void* z, long long z_bs, long long z_ts, int B, int n_rows, int pos0, void* k_cache,
                    void* v_cache, int n_max, unsigned char* ws, const WsLayout& L, CallCtx& ctx) {
  // n_rows positions starting at cache position pos0 (prefill: pos0 = 0; decode: n_rows = 1)
  cudaStream_t s = ctx.s;
  const float scale_log2 = c->softmax_scale * kLog2e;
  PrepassParams pp;
  memset(&pp, 0, sizeof(pp));
  pp.B = B; pp.N = n_rows; pp.d = c->d_model; pp.H = c->n_heads;
  pp.norm_flags = c->norm_flags; pp.eps = c->rms_eps; pp.scale_log2 = scale_log2;
  pp.x = x; pp.x_bs = x_bs; pp.x_ts = x_ts;
  pp.w_q = w->w_q; pp.w_k = w->w_k; pp.w_v = w->w_v;
  pp.g_attn = w->g_attn; pp.g_q = w->g_q; pp.g_k = w->g_k;
  pp.n = ws + L.n; pp.q = ws + L.q; pp.kt = ws + L.kt; pp.vt = ws + L.vt;
  pp.st_o = (float*)(ws + L.st_o); pp.st_m = (float*)(ws + L.st_m); pp.st_l = (float*)(ws + L.st_l);
  pp.sync = (SyncArea*)(ws + L.sync);
  LeafMmaLaunch ml;
  {
    ProfScope ps(s, kProfPrepass);
    if (prepass_launch(c->dtype, pp, s) != cudaSuccess) return RT_ERR_CUDA;
  }

  if (c->recur_block > 1) {
    // Recurrence over blocks of S positions: a block is one parallel sweep (in-block causal attention over the
    // TEMPORARY pairs, the position-wise chain as dense products over the block's rows, then its persistent pairs),
    // and blocks follow each other with Algorithm 1's cross tiles at block granularity.
    if (c->sched != RT_SCHED_TILED || pos0 != 0) return RT_ERR_UNSUPPORTED;
    const int S = c->recur_block, N = n_rows;
    const long long d = c->d_model, f = c->d_ff;
    const size_t e = esize_of(c->dtype);
    SyncArea* sync = (SyncArea*)(ws + L.sync);
    const bool pre = (c->norm_flags & RT_NORM_PRE) != 0;
    TileParams tp;
    memset(&tp, 0, sizeof(tp));
    tp.B = B; tp.d = c->d_model; tp.H = c->n_heads; tp.scale_log2 = scale_log2; tp.alibi = w->alibi_slopes;
    tp.q = ws + L.q; tp.st_o = pp.st_o; tp.st_m = pp.st_m; tp.st_l = pp.st_l;
    tp.rows_q = n_rows; tp.sync = sync;
    PrepassParams pk = pp;                                      // persistent pairs of a block from its outputs
    pk.x_bs = z_bs; pk.x_ts = z_ts;
    pk.norm_flags = (c->norm_flags & RT_NORM_SKIP_Z) ? (c->norm_flags & ~RT_NORM_PRE) : c->norm_flags;
    pk.g_attn = w->g_kv ? w->g_kv : w->g_attn;
    pk.mats = 6; pk.no_seed = 1; pk.chained = 1;              // the chain of a block: programmatic dependent launches
    DenseParams dp;
    memset(&dp, 0, sizeof(dp));
    dp.chained = 1;
    dp.B = B; dp.alpha = c->residual_scale; dp.h = (float*)(ws + L.blk_h);
    const int Lb = c->dtype == RT_BF16 ? 2 * kAutoLeaf : kAutoLeaf;
    for (int s0 = 0; s0 < N; s0 += S) {
      const int e0 = s0 + S < N ? s0 + S : N, rows = e0 - s0;
      {
        // 1. in-block attention over the temporary pairs of strictly earlier positions (the pair of the position
        //    itself is in the seeded state): causal diagonal blocks, then the levels inside the block
        ProfScope ps(s, kProfTile);
        tp.k_cache = ws + L.kt; tp.v_cache = ws + L.vt; tp.rows_kv = n_rows; tp.q_limit = e0;
        const int full = rows / Lb;
        tp.causal = 1;
        if (c->dtype == RT_BF16 && rows % Lb == 0 && rows >= 4 * Lb) {
          // whole blocks of 128, tensor cores: every query's causal prefix inside the block in one launch
          tp.q0 = s0; tp.q1 = e0; tp.k0 = s0; tp.k1 = e0; tp.batch = 0; tp.batch_stride = 0; tp.causal_full = 1;
          if (tile_launch(c->dtype, tp, s) != cudaSuccess) return RT_ERR_CUDA;
          tp.causal_full = 0;
        } else {
          if (full > 0) {
            tp.q0 = s0; tp.q1 = s0 + Lb; tp.k0 = s0; tp.k1 = s0 + Lb; tp.batch = full; tp.batch_stride = Lb;
            if (tile_launch(c->dtype, tp, s) != cudaSuccess) return RT_ERR_CUDA;
          }
          if (full * Lb < rows) {
            tp.q0 = s0 + full * Lb; tp.q1 = e0; tp.k0 = tp.q0; tp.k1 = e0; tp.batch = 1; tp.batch_stride = 0;
            if (tile_simt_launch(c->dtype, tp, s) != cudaSuccess) return RT_ERR_CUDA;
          }
          tp.causal = 0;
          for (long long P = Lb; P < rows; P *= 2) {
            tp.q0 = s0 + (int)P; tp.q1 = s0 + (int)(2 * P); tp.k0 = s0; tp.k1 = s0 + (int)P;
            tp.batch = (int)((rows - P + 2 * P - 1) / (2 * P)); tp.batch_stride = (int)(2 * P);
            if (tile_launch(c->dtype, tp, s) != cudaSuccess) return RT_ERR_CUDA;
          }
        }
        tp.causal = 0; tp.batch = 0; tp.batch_stride = 0; tp.q_limit = 0;
      }
      {
        // 2. position-wise chain over the block's rows, 3. its persistent pairs
        ProfScope ps(s, kProfLeaf);
        const size_t row = (size_t)s0 * B;
        void* cbuf = ws + L.blk_c; void* ubuf = ws + L.blk_u; void* gbuf = ws + L.blk_g;
        if (attn_value_launch(c->dtype, pp.st_o + row * d, pp.st_l + row * c->n_heads, cbuf, (long long)rows * B, (int)d, c->n_heads, s, true) != cudaSuccess)
          return RT_ERR_CUDA;
        dp.M = rows * B;
        dp.N = (int)d; dp.K = (int)d; dp.A = cbuf; dp.W = w->w_o; dp.epi = DENSE_RES_X;
        dp.x = (const unsigned char*)x + (size_t)s0 * x_ts * e; dp.x_bs = x_bs; dp.x_ts = x_ts;
        if (dense_launch(c->dtype, dp, sync, s) != cudaSuccess) return RT_ERR_CUDA;
        if (rms_rows_f32_launch(c->dtype, dp.h, w->g_mlp, ubuf, rows * B, (int)d, c->rms_eps, pre ? 1 : 0, s, true) != cudaSuccess) return RT_ERR_CUDA;
        dp.N = (int)f; dp.K = (int)d; dp.A = ubuf; dp.W = w->w_up; dp.epi = DENSE_GELU; dp.out = gbuf;
        if (dense_launch(c->dtype, dp, sync, s) != cudaSuccess) return RT_ERR_CUDA;
        dp.N = (int)d; dp.K = (int)f; dp.A = gbuf; dp.W = w->w_down; dp.epi = DENSE_RES_H;
        dp.out = (unsigned char*)z + (size_t)s0 * z_ts * e; dp.o_bs = z_bs; dp.o_ts = z_ts;
        if (dense_launch(c->dtype, dp, sync, s) != cudaSuccess) return RT_ERR_CUDA;
        pk.N = rows;
        pk.x = (const unsigned char*)z + (size_t)s0 * z_ts * e;
        pk.kt = (unsigned char*)k_cache + row * d * e; pk.vt = (unsigned char*)v_cache + row * d * e;
        if (prepass_launch(c->dtype, pk, s) != cudaSuccess) return RT_ERR_CUDA;
      }
      if (e0 < N) {
        // 4. Algorithm 1 at block granularity: the next P positions attend to the last P persistent pairs
        const int u = e0 / S;
        const long long P = (long long)S * (u & -u);
        tp.k_cache = k_cache; tp.v_cache = v_cache; tp.rows_kv = n_max;
        tp.q0 = e0; tp.q1 = e0 + P < N ? (int)(e0 + P) : N; tp.k0 = (int)(e0 - P); tp.k1 = e0;
        ProfScope ps(s, kProfTile);
        if (tile_launch(c->dtype, tp, s) != cudaSuccess) return RT_ERR_CUDA;
      }
    }
    return RT_OK;
  }

  const Schedule plan = effective_schedule(c, B, n_rows);
  const bool wide = plan.path == kPathWide && pos0 == 0;
  if (wide) {
    // Wide batches (the regime of the paper's own experiments, Sec. 6: B in the hundreds): a token step is a chain
    // of dense products with M = B rows, so it runs on the tensor cores through the same kernels as the parallel
    // sweep, one position at a time; the schedule (leaf, then the cross tile of Algorithm 1) is unchanged.
    if (c->sched != RT_SCHED_TILED || pos0 != 0) return RT_ERR_UNSUPPORTED;
    const long long d = c->d_model, f = c->d_ff;
    const size_t e = esize_of(c->dtype);
    SyncArea* sync = (SyncArea*)(ws + L.sync);
    float* hbuf = (float*)(ws + L.ex_h);                        // [B, d] fp32
    void* gbuf = ws + L.ex_g;                                   // [B, d_ff] storage type
    void* ubuf = ws + L.ex_z;                                   // [B, d] storage type
    void* cbuf = ws + L.ex_k;                                   // [B, d] storage type
    const bool pre = (c->norm_flags & RT_NORM_PRE) != 0;
    TileParams tp;
    memset(&tp, 0, sizeof(tp));
    tp.B = B; tp.d = c->d_model; tp.H = c->n_heads; tp.scale_log2 = scale_log2; tp.alibi = w->alibi_slopes;
    tp.q = ws + L.q; tp.k_cache = k_cache; tp.v_cache = v_cache;
    tp.st_o = pp.st_o; tp.st_m = pp.st_m; tp.st_l = pp.st_l;
    tp.rows_q = n_rows; tp.rows_kv = n_max; tp.sync = sync;
    PrepassParams pk = pp;                                      // persistent pair of one position from its output
    pk.N = 1; pk.x_bs = z_bs; pk.x_ts = z_ts;
    pk.norm_flags = (c->norm_flags & RT_NORM_SKIP_Z) ? (c->norm_flags & ~RT_NORM_PRE) : c->norm_flags;
    pk.g_attn = w->g_kv ? w->g_kv : w->g_attn;
    pk.mats = 6; pk.no_seed = 1;
    // the seven launches of a token step are short and strictly dependent: chained (programmatic dependent
    // launches), each is scheduled while its predecessor drains
    pk.chained = 1; tp.chained = 1;
    DenseParams dp;
    memset(&dp, 0, sizeof(dp));
    dp.chained = 1;
    dp.M = B; dp.B = B; dp.alpha = c->residual_scale; dp.h = hbuf;
    dp.partial = (float*)(ws + L.ex_part); dp.partial_bytes = (size_t)B * c->n_heads * kMaxChunks * 68 * 4;
    // in-leaf attention re-reads the leaf's pairs for every position (leaf^2 * B * d bytes per leaf), so wide
    // batches default to a shorter leaf
    const int Lf = plan.leaf, N = n_rows;
    // one launch per leaf where the shape allows (rt_wide_loop.cu), else the launches of every position
    const bool loop = c->dtype == RT_BF16 && wide_loop_groups(B, c->d_model, c->d_ff) > 0 && x_bs % 8 == 0 && x_ts % 8 == 0 && z_bs % 8 == 0 && z_ts % 8 == 0;
    WideFwdParams wf;
    memset(&wf, 0, sizeof(wf));
    if (loop) {
      // counters and the bf16 operand rows live in the unused halves of the exchange buffers
      wf.B = B; wf.d = (int)d; wf.H = c->n_heads; wf.dff = (int)f; wf.norm_flags = c->norm_flags; wf.eps = c->rms_eps; wf.scale_log2 = scale_log2; wf.alpha = c->residual_scale;
      wf.w_o = w->w_o; wf.w_up = w->w_up; wf.w_down = w->w_down; wf.w_k = w->w_k; wf.w_v = w->w_v;
      wf.g_mlp = w->g_mlp; wf.g_kv = w->g_kv ? w->g_kv : w->g_attn; wf.g_k = w->g_k; wf.alibi = w->alibi_slopes;
      wf.x = x; wf.x_bs = x_bs; wf.x_ts = x_ts; wf.z = z; wf.z_bs = z_bs; wf.z_ts = z_ts;
      wf.q = ws + L.q; wf.st_o = pp.st_o; wf.st_m = pp.st_m; wf.st_l = pp.st_l; wf.k_cache = k_cache; wf.v_cache = v_cache;
      wf.h = hbuf; wf.partial = dp.partial; wf.c16 = cbuf; wf.u16 = ubuf; wf.g16 = gbuf; wf.r16 = ws + L.ex_z + (size_t)B * d * 2;
      wf.ssq_h = (float*)(ws + L.ex_k + (size_t)B * d * 2);
      wf.counters = (unsigned*)(ws + L.ex_g + align_up((size_t)B * f * 2, 256)); wf.sync = sync;
      if (cudaMemsetAsync(wf.counters, 0, wide_counter_bytes(B), s) != cudaSuccess) return RT_ERR_CUDA;
    }
    for (int s0 = 0; s0 < N; s0 += Lf) {
      const int e0 = s0 + Lf < N ? s0 + Lf : N;
      if (loop) {
        ProfScope ps(s, kProfLeaf);
        wf.t0 = s0; wf.t1 = e0; wf.steps = (unsigned)s0;
        if (wide_forward_launch(wf, s) != cudaSuccess) return RT_ERR_CUDA;
      } else {
        ProfScope ps(s, kProfLeaf);
        for (int t = s0; t < e0; ++t) {
          // pairs of this leaf revealed so far (none for its first position), then c = o / l of the finished row
          tp.q0 = t; tp.q1 = t + 1; tp.k0 = s0; tp.k1 = t; tp.c_out = cbuf;
          if (row_attn_launch(c->dtype, tp, s) != cudaSuccess) return RT_ERR_CUDA;
          tp.c_out = nullptr;
          const size_t row = (size_t)t * B;
          bool normed = false;
          dp.N = (int)d; dp.K = (int)d; dp.A = cbuf; dp.W = w->w_o; dp.epi = DENSE_RES_X;
          dp.x = (const unsigned char*)x + (size_t)t * x_ts * e; dp.x_bs = x_bs; dp.x_ts = 0;
          dp.norm_out = ubuf; dp.norm_gain = w->g_mlp; dp.norm_eps = c->rms_eps; dp.norm_pre = pre ? 1 : 0;   // u = RMS(h)
          if (dense_launch(c->dtype, dp, sync, s, &normed) != cudaSuccess) return RT_ERR_CUDA;
          if (!normed && rms_rows_f32_launch(c->dtype, hbuf, w->g_mlp, ubuf, B, (int)d, c->rms_eps, pre ? 1 : 0, s, true) != cudaSuccess)
            return RT_ERR_CUDA;
          dp.norm_out = nullptr;
          dp.N = (int)f; dp.K = (int)d; dp.A = ubuf; dp.W = w->w_up; dp.epi = DENSE_GELU; dp.out = gbuf;
          if (dense_launch(c->dtype, dp, sync, s) != cudaSuccess) return RT_ERR_CUDA;
          dp.N = (int)d; dp.K = (int)f; dp.A = gbuf; dp.W = w->w_down; dp.epi = DENSE_RES_H;
          dp.out = (unsigned char*)z + (size_t)t * z_ts * e; dp.o_bs = z_bs; dp.o_ts = 0;
          dp.norm_out = pk.n; dp.norm_gain = pk.g_attn; dp.norm_pre = (pk.norm_flags & RT_NORM_PRE) ? 1 : 0;          // RMS(z)
          if (dense_launch(c->dtype, dp, sync, s, &normed) != cudaSuccess) return RT_ERR_CUDA;
          dp.norm_out = nullptr;
          pk.skip_rms = normed ? 1 : 0;
          pk.x = (const unsigned char*)z + (size_t)t * z_ts * e;
          pk.kt = (unsigned char*)k_cache + row * d * e; pk.vt = (unsigned char*)v_cache + row * d * e;
          if (prepass_launch(c->dtype, pk, s) != cudaSuccess) return RT_ERR_CUDA;
        }
      }
      if (e0 < N) {
        const int P = e0 & -e0;
        tp.q0 = e0; tp.q1 = e0 + P < N ? e0 + P : N; tp.k0 = e0 - P; tp.k1 = e0;
        ProfScope ps(s, kProfTile);
        if (tile_launch(c->dtype, tp, s) != cudaSuccess) return RT_ERR_CUDA;
      }
    }
    return RT_OK;
  }

  LeafLaunch ll;
  if (leaf_plan(c->dtype, B, c->d_model, c->d_ff, &ll) != cudaSuccess) return RT_ERR_CUDA;
  LeafParams lp;
  memset(&lp, 0, sizeof(lp));
  lp.B = B; lp.d = c->d_model; lp.H = c->n_heads; lp.dff = c->d_ff;
  lp.norm_flags = c->norm_flags; lp.eps = c->rms_eps; lp.scale_log2 = scale_log2; lp.alpha = c->residual_scale;
  lp.w_o = w->w_o; lp.w_up = w->w_up; lp.w_down = w->w_down; lp.w_k = w->w_k; lp.w_v = w->w_v;
  lp.g_mlp = w->g_mlp; lp.g_kv = w->g_kv ? w->g_kv : w->g_attn; lp.g_k = w->g_k; lp.alibi = w->alibi_slopes;
  lp.x = x; lp.x_bs = x_bs; lp.x_ts = x_ts;
  lp.z = z; lp.z_bs = z_bs; lp.z_ts = z_ts;
  lp.k_cache = k_cache; lp.v_cache = v_cache;
  lp.q = ws + L.q;
  lp.st_o = pp.st_o; lp.st_m = pp.st_m; lp.st_l = pp.st_l;
  lp.row_off = pos0;
  lp.ex_h = (float*)(ws + L.ex_h); lp.ex_g = (float*)(ws + L.ex_g);
  lp.ex_z = (float*)(ws + L.ex_z); lp.ex_k = (float*)(ws + L.ex_k);
  lp.ex_part = (float*)(ws + L.ex_part);
  lp.max_chunks = kMaxChunks;
  lp.timers = g_prof_timers ? 1 : 0;
  lp.sync = (SyncArea*)(ws + L.sync);

  // small layers: the whole chain inside one cluster, same leaves and tiles
  LeafSmallLaunch sl;
  const bool small = c->sched == RT_SCHED_TILED && pos0 == 0 &&
                     leaf_small_shape(c->dtype, B, c->d_model, c->n_heads, c->d_ff, plan.leaf, kB200SmemPerCta, &sl);
  auto leaf = [&](int t0, int t1, int attn_begin) -> bool {
    lp.t0 = t0; lp.t1 = t1; lp.attn_begin = attn_begin; lp.bar_base = ctx.bar_base;
    ProfScope ps(s, kProfLeaf);
    if (leaf_launch(c->dtype, lp, ll, s) != cudaSuccess) return false;
    ctx.bar_base += leaf_barrier_arrivals(t0, t1, ll.grid);
    return true;
  };

  // bf16 tiled prefill takes the tensor-core leaf kernel when the shape fits it
  // (batches of 17 .. 48 sequences: in slices of at most 16, see effective_schedule)
  const int b_sub = (plan.path == kPathMmaSplit && pos0 == 0) ? plan.sub : B;
  const bool use_mma = !small && c->dtype == RT_BF16 && c->sched == RT_SCHED_TILED && pos0 == 0 &&
                       leaf_mma_plan(b_sub, c->d_model, c->n_heads, c->d_ff, c->leaf, &ml);
  LeafMmaBuffers mb;
  mb.vectors = nullptr; mb.ll_kv = (unsigned long long*)(ws + L.ll);
  auto leaf_mma = [&](int t0, int t1) -> bool {
    ProfScope ps(s, kProfLeaf);
    const size_t e = esize_of(c->dtype);
    for (int b0 = 0; b0 < B; b0 += b_sub) {
      lp.B = B - b0 < b_sub ? B - b0 : b_sub; lp.Bs = B; lp.b0 = b0;
      lp.x = (const unsigned char*)x + (size_t)b0 * x_bs * e;
      lp.z = (unsigned char*)z + (size_t)b0 * z_bs * e;
      lp.t0 = t0; lp.t1 = t1; lp.attn_begin = t0; lp.seq_base = ctx.seq_base;
      // fresh arrays of c, h, z and g for the positions of this launch; filled all at once when they run out
      const size_t set_bytes = leaf_mma_set_bytes(c->d_model, c->d_ff);
      if (ctx.sets_left < t1 - t0) {
        if (cudaMemsetAsync(ws + L.form, 0xff, L.sets * set_bytes, s) != cudaSuccess) return false;
        ctx.sets_left = (int)L.sets;
      }
      mb.vectors = ws + L.form + (L.sets - (size_t)ctx.sets_left) * set_bytes;
      ctx.sets_left -= t1 - t0;
      if (leaf_mma_launch(lp, ml, mb, s) != cudaSuccess) return false;
      ctx.seq_base += (unsigned)(t1 - t0);
    }
    return true;
  };

  if (c->sched == RT_SCHED_NAIVE || pos0 > 0) {
    // token-sequential: every position reads its whole prefix from the cache
    return leaf(pos0, pos0 + n_rows, 0) ? RT_OK : RT_ERR_CUDA;
  }
  TileParams tp;
  memset(&tp, 0, sizeof(tp));
  tp.B = B; tp.d = c->d_model; tp.H = c->n_heads; tp.scale_log2 = scale_log2; tp.alibi = w->alibi_slopes;
  tp.q = ws + L.q; tp.k_cache = k_cache; tp.v_cache = v_cache;
  tp.st_o = pp.st_o; tp.st_m = pp.st_m; tp.st_l = pp.st_l;
  tp.rows_q = n_rows; tp.rows_kv = n_max; tp.sync = lp.sync;
  auto leaf_small = [&](int t0, int t1) -> bool {
    lp.t0 = t0; lp.t1 = t1; lp.attn_begin = t0;
    ProfScope ps(s, kProfLeaf);
    return leaf_small_launch(c->dtype, lp, sl, s) == cudaSuccess;
  };
  const bool groups = !small && plan.path == kPathGroups && pos0 == 0;
  const int places = groups ? ceil_div(B, plan.sub) : 0;
  unsigned char* const packed = groups ? ws + L.form + group_area(c, places, 1, 0, 0).packed : nullptr;
  if (groups) {
    if (!clear_groups(c, places, ws, L, ctx)) return RT_ERR_CUDA;
    const GroupPackLayer pl = {w->w_o, w->w_up, w->w_down, w->w_k, w->w_v, packed};
    ProfScope ps(s, kProfPrepass);
    if (leaf_group_pack(&pl, 1, c->d_model, c->d_ff, places, s) != cudaSuccess) return RT_ERR_CUDA;
  }
  auto leaf_groups = [&](int t0, int t1) -> bool {
    ProfScope ps(s, kProfLeaf);
    const size_t e = esize_of(c->dtype);
    GroupJob jobs[kGroupJobs];
    memset(jobs, 0, sizeof(jobs));
    for (int i = 0; i < places; ++i) {
      GroupJob& j = jobs[i];
      const int b0 = i * plan.sub;
      j.packed = packed; j.g_mlp = lp.g_mlp; j.g_kv = lp.g_kv; j.g_k = lp.g_k; j.alibi = w->alibi_slopes;
      j.q = lp.q; j.st_o = lp.st_o; j.st_m = lp.st_m; j.st_l = lp.st_l; j.row_off = 0;
      j.x = (const unsigned char*)x + (size_t)b0 * x_bs * e; j.x_bs = x_bs; j.x_ts = x_ts;
      j.z = (unsigned char*)z + (size_t)b0 * z_bs * e; j.z_bs = z_bs; j.z_ts = z_ts;
      j.k_cache = k_cache; j.v_cache = v_cache; j.t0 = t0; j.t1 = t1; j.key0 = t0;
      j.B = B - b0 < plan.sub ? B - b0 : plan.sub; j.b0 = b0;
      j.words = ws + L.form + (size_t)i * leaf_group_words_bytes(c->d_model, c->d_ff); j.steps = ctx.group_steps[i];
      ctx.group_steps[i] += (unsigned)(t1 - t0);
    }
    return leaf_group_launch(group_common(c, B, ws, L), jobs, places, places, s) == cudaSuccess;
  };
  const int Lf = groups ? plan.leaf : small ? sl.leaf : (use_mma ? ml.leaf : leaf_size(c)), N = n_rows;
  for (int s0 = 0; s0 < N; s0 += Lf) {
    const int e0 = s0 + Lf < N ? s0 + Lf : N;
    if (!(groups ? leaf_groups(s0, e0) : small ? leaf_small(s0, e0) : (use_mma ? leaf_mma(s0, e0) : leaf(s0, e0, s0)))) return RT_ERR_CUDA;
    if (e0 < N) {
      const int P = e0 & -e0;                              // largest power of two dividing the block end
      tp.q0 = e0; tp.q1 = e0 + P < N ? e0 + P : N; tp.k0 = e0 - P; tp.k1 = e0;
      ProfScope ps(s, kProfTile);
      if ((wave_exact_tile(ctx.exact, e0) && P % kWaveBlock == 0 ? tile_rows_batch_launch(&tp, 1, s) : tile_launch(c->dtype, tp, s)) != cudaSuccess) return RT_ERR_CUDA;
    }
  }
  return RT_OK;
}

// Whether any two caches share rows.  Layers one after the other may (a program that wants the logits only can give every layer the same
// pair); side by side they write their rows at the same time.
bool caches_overlap(const rt_config* c, int n_layers, int B, int N, void* const* k_caches, void* const* v_caches) {
  const size_t bytes = (size_t)N * B * c->d_model * esize_of(c->dtype);
  for (int i = 0; i < 2 * n_layers; ++i)
    for (int j = 0; j < i; ++j)
      if (overlaps(i < n_layers ? k_caches[i] : v_caches[i - n_layers], bytes, j < n_layers ? k_caches[j] : v_caches[j - n_layers], bytes)) return true;
  return false;
}

// All layers of a stack, several at a time (stack_wave): x^0 in hid[0], layer l reads hid[l & 1] and writes hid[(l + 1) & 1] (the
// last one `out`, if given); a row is overwritten only after the layer that reads it has finished it.
rt_status run_stack_wave(const rt_config* c, int n_layers, const rt_layer_weights* layers, void* const* hid, void* out, int B, int N, void* const* k_caches,
                         void* const* v_caches, int N_max, unsigned char* ws, const WsLayout& L, const Wave& wv, CallCtx& ctx) {
  cudaStream_t s = ctx.s;
  const int places = wv.places, n_leaves = ceil_div(N, wv.leaf), bands = ceil_div(n_layers, wv.packs);
  const size_t e = esize_of(c->dtype), d = c->d_model;
  const WaveRows W = wave_rows_layout(c, B, wv.leaf);
  const GroupArea A = group_area(c, places, wv.packs, B, wv.leaf);
  if (!clear_groups(c, places, ws, L, ctx)) return RT_ERR_CUDA;
  auto packed = [&](int l) { return ws + L.form + A.packed + (size_t)l * A.packed_stride; };
  const GroupCommon gc = group_common(c, B, ws, L);
  const long long bs = (long long)N * d;
  for (int b = 0; b < bands; ++b) {
    const int l0 = band_begin(n_layers, bands, b), band = band_begin(n_layers, bands, b + 1) - l0;
    {
      ProfScope ps(s, kProfPrepass);
      for (int i = 0; i < band; i += kGroupPackLayers) {
        GroupPackLayer pl[kGroupPackLayers];
        const int here = band - i < kGroupPackLayers ? band - i : kGroupPackLayers;
        for (int k = 0; k < here; ++k) {
          const rt_layer_weights& w = layers[l0 + i + k];
          pl[k] = {w.w_o, w.w_up, w.w_down, w.w_k, w.w_v, packed(i + k)};
        }
        if (leaf_group_pack(pl, here, c->d_model, c->d_ff, places, s) != cudaSuccess) return RT_ERR_CUDA;
      }
    }
    WaveOrder order(band, n_leaves);
    int of[kGroupJobs], leaf_of[kGroupJobs];
    for (int nj; (nj = order.next(places, of, leaf_of)) > 0;) {
      GroupJob jobs[kGroupJobs];
      PrepassParams pre[kGroupJobs];
      memset(jobs, 0, sizeof(jobs));
      memset(pre, 0, sizeof(pre));
      for (int i = 0; i < nj; ++i) {
        const int l = l0 + of[i], t0 = leaf_of[i] * wv.leaf, t1 = t0 + wv.leaf < N ? t0 + wv.leaf : N;
        const rt_layer_weights& w = layers[l];
        unsigned char* rows = ws + L.form + A.rows + A.rows_stride * i;
        PrepassParams& pp = pre[i];
        pp.B = B; pp.N = t1 - t0; pp.d = c->d_model; pp.H = c->n_heads; pp.norm_flags = c->norm_flags; pp.eps = c->rms_eps; pp.scale_log2 = gc.scale_log2;
        pp.x = (const unsigned char*)hid[l & 1] + (size_t)t0 * d * e; pp.x_bs = bs; pp.x_ts = (long long)d;
        pp.w_q = w.w_q; pp.w_k = w.w_k; pp.w_v = w.w_v; pp.g_attn = w.g_attn; pp.g_q = w.g_q; pp.g_k = w.g_k;
        pp.n = rows + W.n; pp.q = rows + W.q; pp.kt = rows + W.kt; pp.vt = rows + W.vt;
        pp.st_o = (float*)(rows + W.st_o); pp.st_m = (float*)(rows + W.st_m); pp.st_l = (float*)(rows + W.st_l); pp.sync = gc.sync;
        GroupJob& j = jobs[i];
        j.packed = packed(of[i]); j.g_mlp = w.g_mlp; j.g_kv = w.g_kv ? w.g_kv : w.g_attn; j.g_k = w.g_k; j.alibi = w.alibi_slopes;
        j.q = pp.q; j.st_o = pp.st_o; j.st_m = pp.st_m; j.st_l = pp.st_l; j.row_off = t0;
        j.x = hid[l & 1]; j.x_bs = bs; j.x_ts = (long long)d;
        j.z = l == n_layers - 1 && out ? out : hid[(l + 1) & 1]; j.z_bs = bs; j.z_ts = (long long)d;
        j.k_cache = k_caches[l]; j.v_cache = v_caches[l]; j.t0 = t0; j.t1 = t1; j.B = B; j.b0 = 0;
        j.key0 = t0 / kWaveBlock * kWaveBlock;
        j.words = ws + L.form + (size_t)i * leaf_group_words_bytes(c->d_model, c->d_ff); j.steps = ctx.group_steps[i];
        ctx.group_steps[i] += (unsigned)(t1 - t0);
      }
      {
        ProfScope ps(s, kProfPrepass);
        if (prepass_batch_launch(c->dtype, pre, nj, s) != cudaSuccess) return RT_ERR_CUDA;
      }
      // The leaf's queries against the whole blocks of kWaveBlock earlier pairs; the kernel absorbs the rest.
      TileParams tiles[kGroupJobs];
      // (distances alone, without a scale, are not for the tensor-core tile either)
      auto fp32_tile = [&](int i) { return wave_exact_tile(wv.exact, jobs[i].t0) || (jobs[i].alibi && gc.scale_log2 == 0.f); };
      auto tile_of = [&](int i, int k0, int k1) {
        TileParams tp;
        memset(&tp, 0, sizeof(tp));
        tp.B = B; tp.d = c->d_model; tp.H = c->n_heads; tp.scale_log2 = gc.scale_log2; tp.alibi = jobs[i].alibi;
        tp.q = pre[i].q; tp.k_cache = jobs[i].k_cache; tp.v_cache = jobs[i].v_cache; tp.st_o = pre[i].st_o; tp.st_m = pre[i].st_m; tp.st_l = pre[i].st_l;
        tp.rows_q = pre[i].N; tp.rows_kv = N_max; tp.sync = gc.sync; tp.q_pos0 = jobs[i].t0;
        tp.q0 = 0; tp.q1 = pre[i].N; tp.k0 = k0; tp.k1 = k1;
        return tp;
      };
      {
        int nt = 0;
        for (int i = 0; i < nj; ++i)
          if (jobs[i].key0 && fp32_tile(i)) tiles[nt++] = tile_of(i, 0, jobs[i].key0);
        if (nt) {
          ProfScope ps(s, kProfTile);
          if (tile_rows_batch_launch(tiles, nt, s) != cudaSuccess) return RT_ERR_CUDA;
        }
      }
      // On tensor cores they come in the parts in which Algorithm 1's tiles would have brought them (the powers of two that the number of blocks
      // consists of, largest first): the same states to the bit.
      for (int part = 0, more = 1; more; ++part) {
        more = 0;
        for (int sloped = 0; sloped < 2; ++sloped) {
          int nt = 0;
          for (int i = 0; i < nj; ++i) {
            int blocks = fp32_tile(i) ? 0 : jobs[i].key0 / kWaveBlock, k0 = 0, size = 0;
            for (int skip = 0; blocks && skip <= part; ++skip) {
              k0 += size;
              size = 1;
              while (size * 2 <= blocks) size *= 2;
              blocks -= size;
              if (skip == part) {
                more |= blocks > 0;
                if ((jobs[i].alibi != nullptr) != (sloped != 0)) break;
                tiles[nt++] = tile_of(i, k0 * kWaveBlock, (k0 + size) * kWaveBlock);
              }
            }
          }
          if (!nt) continue;
          ProfScope ps(s, kProfTile);
          if (tile_tc_batch_launch(tiles, nt, gc.sync, s) != cudaSuccess) return RT_ERR_CUDA;
        }
      }
      ProfScope ps(s, kProfLeaf);
      if (leaf_group_launch(gc, jobs, nj, places, s) != cudaSuccess) return RT_ERR_CUDA;
    }
  }
  return RT_OK;
}

// Whether the vectors between the phases of a decode step stay fp32: wherever the generic leaf kernel would answer otherwise, which holds
// them so (batches above 16, a first position, layers off the tensor-core leaf kernel).  The error of the appended k, v rows against 64 bits is
// 3.5e-3 that way and 4.1e-3 with bf16 vectors (d = 1024, 8 layers, 512 positions), for d = 2048 2.0e-3 and 2.9e-3.
bool decode_full(const rt_config* c, int B, int pos) {
  LeafMmaLaunch ml;
  return B > 16 || pos == 0 || !leaf_mma_shape(B, c->d_model, c->n_heads, c->d_ff, c->leaf, kB200Sms, kB200SmemPerCta, &ml);
}

// One decode step through all layers on the decode kernel (bf16): slices of at most 16 (fp32 vectors: 8) sequences, launches of at most
// kDecMaxLayers layers.  Input rows x (row stride x_bs) or embedding rows emb[ids]; output rows z.  `hid` holds [B, d] rows between launches.
rt_status run_decode(const rt_config* c, int n_layers, const rt_layer_weights* layers, const void* x, long long x_bs, const void* emb,
                     const int32_t* ids, int vocab, int B, int pos, void* z, long long z_bs, void* const* k_caches, void* const* v_caches,
                     unsigned char* ws, const WsLayout& L, void* const* hid, const void* next_bytes, size_t next_size, cudaStream_t s) {
  const bool full = decode_full(c, B, pos);
  const int sub = decode_slice(B, full), d = c->d_model;
  ProfScope ps(s, kProfLeaf);
  for (int b0 = 0; b0 < B; b0 += sub) {
    DecodeParams p;
    memset(&p, 0, sizeof(p));
    p.B = B - b0 < sub ? B - b0 : sub; p.Bs = B; p.b0 = b0;
    p.d = d; p.H = c->n_heads; p.dff = c->d_ff; p.pos = pos; p.full = full ? 1 : 0;
    p.norm_flags = c->norm_flags; p.eps = c->rms_eps; p.scale_log2 = c->softmax_scale * kLog2e; p.alpha = c->residual_scale;
    p.words = ws + L.dec_words; p.words_size = L.dec_words_bytes; p.sync = (SyncArea*)(ws + L.sync);
    for (int l0 = 0; l0 < n_layers; l0 += kDecMaxLayers) {
      const bool to_z = l0 + kDecMaxLayers >= n_layers;
      const size_t off = (size_t)b0 * 2;
      p.n_layers = to_z ? n_layers - l0 : kDecMaxLayers;
      p.x = nullptr; p.ids = nullptr;
      if (l0 > 0) { p.x = (const unsigned char*)hid[(l0 / kDecMaxLayers - 1) & 1] + off * d; p.x_bs = d; }
      else if (x) { p.x = (const unsigned char*)x + off * x_bs; p.x_bs = x_bs; }
      else { p.emb = emb; p.ids = ids + b0; p.vocab = vocab; }
      p.z_out = (unsigned char*)(to_z ? z : hid[(l0 / kDecMaxLayers) & 1]) + off * (to_z ? z_bs : d);
      p.z_bs = to_z ? z_bs : d;
      if (to_z && b0 + sub >= B) { p.next_bytes = next_bytes; p.next_size = next_size; }
      for (int l = 0; l < p.n_layers; ++l) {
        const rt_layer_weights& w = layers[l0 + l];
        DecLayer& o = p.layer[l];
        o.w_q = w.w_q; o.w_k = w.w_k; o.w_v = w.w_v; o.w_o = w.w_o; o.w_up = w.w_up; o.w_down = w.w_down;
        o.g_attn = w.g_attn; o.g_mlp = w.g_mlp; o.g_kv = w.g_kv ? w.g_kv : w.g_attn; o.g_q = w.g_q; o.g_k = w.g_k;
        o.alibi = w.alibi_slopes; o.k_cache = k_caches[l0 + l]; o.v_cache = v_caches[l0 + l];
      }
      if (decode_launch(p, s) != cudaSuccess) return RT_ERR_CUDA;
    }
  }
  return RT_OK;
}

// bf16 shapes that the decode kernel takes; everything else takes the generic leaf kernel.
bool decode_fast(const rt_config* c, int B) { return c->dtype == RT_BF16 && decode_shape(B, c->d_model, c->n_heads, c->d_ff); }

rt_status common_checks(const rt_config* c, int B, int N, int n_layers, void* ws, size_t ws_bytes, bool wide_ok = false) {      // n_layers: that the workspace has to suffice for
  if (!config_ok(c) || B <= 0 || N <= 0 || n_layers <= 0 || !ws || !aligned16(ws)) return RT_ERR_INVALID_ARG;
  const rt_status st = config_supported(c, B, wide_ok);
  if (st != RT_OK) return st;
  // the recurrence over blocks exists for tiled prefill only (wide_ok marks the prefill entry points)
  if (c->recur_block > 1 && !(wide_ok && c->sched == RT_SCHED_TILED)) return RT_ERR_UNSUPPORTED;
  if (ws_bytes < ws_layout(c, B, N, n_layers).total) return RT_ERR_WORKSPACE;
  return RT_OK;
}

}  // namespace

namespace rt {
ProfSpanScope::ProfSpanScope(cudaStream_t s, int cls) { impl = new ProfScope(s, cls); }
ProfSpanScope::~ProfSpanScope() { delete static_cast<ProfScope*>(impl); }
}  // namespace rt

extern "C" {

size_t rt_workspace_bytes(const rt_config* cfg, int32_t B, int32_t N, int32_t n_layers) {
  if (!config_ok(cfg) || B <= 0 || N <= 0 || n_layers <= 0) return 0;
  return ws_layout(cfg, B, N, n_layers).total;
}

rt_status rt_layer_prefill(const rt_config* cfg, const rt_layer_weights* w, const void* x, int32_t B, int32_t N,
                           void* z, void* k_cache, void* v_cache, int32_t N_max, void* workspace,
                           size_t workspace_bytes, void* cuda_stream) {
  rt_status st = common_checks(cfg, B, N, 1, workspace, workspace_bytes, true);
  if (st != RT_OK) return st;
  if (!weights_ok(w) || !x || !z || !k_cache || !v_cache || N_max < N) return RT_ERR_INVALID_ARG;
  if (!aligned16(x) || !aligned16(z) || !aligned16(k_cache) || !aligned16(v_cache)) return RT_ERR_INVALID_ARG;
  const size_t xz_bytes = (size_t)B * N * cfg->d_model * esize_of(cfg->dtype);
  if (overlaps(x, xz_bytes, z, xz_bytes)) return RT_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  unsigned char* ws = (unsigned char*)workspace;
  const WsLayout L = ws_layout(cfg, B, N, 1);
  if (cudaMemsetAsync(ws + L.sync, 0, sizeof(SyncArea), s) != cudaSuccess) return RT_ERR_CUDA;
  if (cudaMemsetAsync(ws + L.ll, 0, L.ll_bytes, s) != cudaSuccess) return RT_ERR_CUDA;
  const long long d = cfg->d_model;
  CallCtx ctx{s};
  return run_layer(cfg, w, x, (long long)N * d, d, z, (long long)N * d, d, B, N, 0, k_cache, v_cache, N_max, ws, L, ctx);
}

size_t rt_recompute_workspace_bytes(const rt_config* cfg, int32_t B, int32_t N) {
  if (!config_ok(cfg) || B <= 0 || N <= 0) return 0;
  return ws_layout(cfg, B, N, 1).total + align_up((size_t)B * N * cfg->d_ff * esize_of(cfg->dtype), 256);
}

rt_status rt_layer_recompute(const rt_config* cfg, const rt_layer_weights* w, const void* x, const void* z_claim,
                             int32_t B, int32_t N, void* z_out, void* k_cache, void* v_cache, int32_t N_max,
                             void* workspace, size_t workspace_bytes, void* cuda_stream) {
  if (!config_ok(cfg) || B <= 0 || N <= 0 || !workspace || !aligned16(workspace)) return RT_ERR_INVALID_ARG;
  rt_status st = config_supported(cfg, 1);
  if (st != RT_OK) return st;
  if (cfg->recur_block > 1) return RT_ERR_UNSUPPORTED;          // the sweep is the fixed-point map of the layer of Sec. 2.2
  if (workspace_bytes < rt_recompute_workspace_bytes(cfg, B, N)) return RT_ERR_WORKSPACE;
  if (!weights_ok(w) || !x || !z_claim || !z_out || !k_cache || !v_cache || z_out == x || z_out == z_claim || N_max < N)
    return RT_ERR_INVALID_ARG;
  if (!aligned16(x) || !aligned16(z_claim) || !aligned16(z_out) || !aligned16(k_cache) || !aligned16(v_cache))
    return RT_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  unsigned char* ws = (unsigned char*)workspace;
  const WsLayout L = ws_layout(cfg, B, N, 1);
  if (cudaMemsetAsync(ws + L.sync, 0, sizeof(SyncArea), s) != cudaSuccess) return RT_ERR_CUDA;
  const long long d = cfg->d_model, f = cfg->d_ff;
  const long long tok = (long long)B * N;
  const float scale_log2 = cfg->softmax_scale * kLog2e;
  SyncArea* sync = (SyncArea*)(ws + L.sync);
  const bool pre = (cfg->norm_flags & RT_NORM_PRE) != 0;

  // 1. every persistent pair from the claimed outputs (Eqs. 1-2): k = qkRMS[W_k RMS(z)], v = W_v RMS(z)
  PrepassParams pz;
  memset(&pz, 0, sizeof(pz));
  pz.B = B; pz.N = N; pz.d = cfg->d_model; pz.H = cfg->n_heads;
  pz.norm_flags = (cfg->norm_flags & RT_NORM_SKIP_Z) ? (cfg->norm_flags & ~RT_NORM_PRE) : cfg->norm_flags;
  pz.eps = cfg->rms_eps; pz.scale_log2 = scale_log2;
  pz.x = z_claim; pz.x_bs = (long long)N * d; pz.x_ts = d;
  pz.w_q = w->w_q; pz.w_k = w->w_k; pz.w_v = w->w_v;
  pz.g_attn = w->g_kv ? w->g_kv : w->g_attn; pz.g_q = w->g_q; pz.g_k = w->g_k;
  pz.n = ws + L.n; pz.q = ws + L.q; pz.kt = k_cache; pz.vt = v_cache;
  pz.st_o = (float*)(ws + L.st_o); pz.st_m = (float*)(ws + L.st_m); pz.st_l = (float*)(ws + L.st_l);
  pz.mats = 6; pz.no_seed = 1; pz.sync = sync;
  {
    ProfScope ps(s, kProfPrepass);
    if (prepass_launch(cfg->dtype, pz, s) != cudaSuccess) return RT_ERR_CUDA;
  }
  // 2. queries, temporary pairs and the seeded running stats from the layer input, as in the prefill
  PrepassParams px = pz;
  px.norm_flags = cfg->norm_flags;
  px.x = x; px.g_attn = w->g_attn;
  px.kt = ws + L.kt; px.vt = ws + L.vt;
  px.mats = 0; px.no_seed = 0;
  {
    ProfScope ps(s, kProfPrepass);
    if (prepass_launch(cfg->dtype, px, s) != cudaSuccess) return RT_ERR_CUDA;
  }
  // 3. attention of every query over all earlier persistent pairs: the pairs inside a 64-block under a causal
  //    mask, then Algorithm 1's cross tiles, one launch per level (all pairs are known, so the tiles of a level are
  //    independent; each query row meets exactly one tile per level)
  TileParams tp;
  memset(&tp, 0, sizeof(tp));
  tp.B = B; tp.d = cfg->d_model; tp.H = cfg->n_heads; tp.scale_log2 = scale_log2; tp.alibi = w->alibi_slopes;
  tp.q = ws + L.q; tp.k_cache = k_cache; tp.v_cache = v_cache;
  tp.st_o = px.st_o; tp.st_m = px.st_m; tp.st_l = px.st_l;
  tp.rows_q = N; tp.rows_kv = N_max; tp.sync = sync; tp.q_limit = N;
  {
    ProfScope ps(s, kProfTile);
    // diagonal blocks under the causal mask: whole blocks in one batched launch (tensor cores for bf16), the
    // ragged last block on its own; then the levels of Algorithm 1 from the block size upwards
    const int Lb = cfg->dtype == RT_BF16 ? 2 * kAutoLeaf : kAutoLeaf;
    const int full = N / Lb;
    tp.causal = 1;
    if (cfg->dtype == RT_BF16 && N % Lb == 0 && N >= 4 * Lb) {
      // whole blocks only, tensor cores: every query's causal prefix in ONE launch (a CTA walks over the key blocks up to
      // its own query tile) instead of diagonal blocks plus one launch per level of short tiles
      tp.q0 = 0; tp.q1 = N; tp.k0 = 0; tp.k1 = N; tp.batch = 0; tp.batch_stride = 0; tp.causal_full = 1;
      if (tile_launch(cfg->dtype, tp, s) != cudaSuccess) return RT_ERR_CUDA;
      tp.causal_full = 0; tp.causal = 0;
      goto attention_done;
    }
    if (full > 0) {
      tp.q0 = 0; tp.q1 = Lb; tp.k0 = 0; tp.k1 = Lb; tp.batch = full; tp.batch_stride = Lb;
      if (tile_launch(cfg->dtype, tp, s) != cudaSuccess) return RT_ERR_CUDA;
    }
    if (full * Lb < N) {
      tp.q0 = full * Lb; tp.q1 = N; tp.k0 = full * Lb; tp.k1 = N; tp.batch = 1; tp.batch_stride = 0;
      if (tile_simt_launch(cfg->dtype, tp, s) != cudaSuccess) return RT_ERR_CUDA;
    }
    tp.causal = 0;
    for (long long P = Lb; P < N; P *= 2) {
      tp.q0 = (int)P; tp.q1 = (int)(2 * P); tp.k0 = 0; tp.k1 = (int)P;
      tp.batch = (int)((N - P + 2 * P - 1) / (2 * P)); tp.batch_stride = (int)(2 * P);
      if (tile_launch(cfg->dtype, tp, s) != cudaSuccess) return RT_ERR_CUDA;
    }
  attention_done:;
  }
  // 4. position-wise chain over all rows at once
  ProfScope ps(s, kProfOther);
  void* cbuf = ws + L.kt;                                       // the temporary pairs are folded into the stats by now
  void* ubuf = ws + L.vt;
  float* hbuf = (float*)(ws + L.st_o);                          // free once c = o / l is taken
  void* gbuf = ws + L.total;
  if (attn_value_launch(cfg->dtype, px.st_o, px.st_l, cbuf, tok, (int)d, cfg->n_heads, s) != cudaSuccess) return RT_ERR_CUDA;
  DenseParams dp;
  memset(&dp, 0, sizeof(dp));
  dp.M = (int)tok; dp.B = B; dp.alpha = cfg->residual_scale; dp.h = hbuf;
  dp.N = (int)d; dp.K = (int)d; dp.A = cbuf; dp.W = w->w_o; dp.epi = DENSE_RES_X;
  dp.x = x; dp.x_bs = (long long)N * d; dp.x_ts = d;
  if (dense_launch(cfg->dtype, dp, sync, s) != cudaSuccess) return RT_ERR_CUDA;
  if (rms_rows_f32_launch(cfg->dtype, hbuf, w->g_mlp, ubuf, (int)tok, (int)d, cfg->rms_eps, pre ? 1 : 0, s) != cudaSuccess)
    return RT_ERR_CUDA;
  dp.N = (int)f; dp.K = (int)d; dp.A = ubuf; dp.W = w->w_up; dp.epi = DENSE_GELU; dp.out = gbuf;
  if (dense_launch(cfg->dtype, dp, sync, s) != cudaSuccess) return RT_ERR_CUDA;
  dp.N = (int)d; dp.K = (int)f; dp.A = gbuf; dp.W = w->w_down; dp.epi = DENSE_RES_H;
  dp.out = z_out; dp.o_bs = (long long)N * d; dp.o_ts = d;
  if (dense_launch(cfg->dtype, dp, sync, s) != cudaSuccess) return RT_ERR_CUDA;
  return RT_OK;
}

rt_status rt_layer_decode_step(const rt_config* cfg, const rt_layer_weights* w, const void* x, int32_t B, int32_t pos,
                               void* z, void* k_cache, void* v_cache, int32_t N_max, void* workspace,
                               size_t workspace_bytes, void* cuda_stream) {
  rt_status st = common_checks(cfg, B, 1, 1, workspace, workspace_bytes);
  if (st != RT_OK) return st;
  if (!weights_ok(w) || !x || !z || !k_cache || !v_cache || pos < 0 || pos >= N_max) return RT_ERR_INVALID_ARG;
  if (!aligned16(x) || !aligned16(z) || !aligned16(k_cache) || !aligned16(v_cache)) return RT_ERR_INVALID_ARG;
  {
    const size_t xz_bytes = (size_t)B * cfg->d_model * esize_of(cfg->dtype);
    if (overlaps(x, xz_bytes, z, xz_bytes)) return RT_ERR_INVALID_ARG;
  }
  cudaStream_t s = (cudaStream_t)cuda_stream;
  unsigned char* ws = (unsigned char*)workspace;
  const WsLayout L = ws_layout(cfg, B, 1, 1);
  if (cudaMemsetAsync(ws + L.sync, 0, sizeof(SyncArea), s) != cudaSuccess) return RT_ERR_CUDA;
  const long long d = cfg->d_model;
  if (decode_fast(cfg, B)) {
    void* hid[2] = {ws + L.hid0, ws + L.hid1};
    return run_decode(cfg, 1, w, x, d, nullptr, nullptr, 0, B, pos, z, d, &k_cache, &v_cache, ws, L, hid, nullptr, 0, s);
  }
  if (cudaMemsetAsync(ws + L.ll, 0, L.ll_bytes, s) != cudaSuccess) return RT_ERR_CUDA;
  rt_config c = *cfg;
  c.sched = RT_SCHED_NAIVE;
  CallCtx ctx{s};
  return run_layer(&c, w, x, d, d, z, d, d, B, 1, pos, k_cache, v_cache, N_max, ws, L, ctx);
}

rt_status rt_stack_prefill(const rt_config* cfg, int32_t n_layers, const rt_layer_weights* layers, const void* emb,
                           const void* g_final, int32_t vocab, const int32_t* ids, int32_t B, int32_t N, void* hidden,
                           float* logits_last, void* const* k_caches, void* const* v_caches, int32_t N_max,
                           void* workspace, size_t workspace_bytes, void* cuda_stream) {
  if (n_layers <= 0) return RT_ERR_INVALID_ARG;
  rt_status st = common_checks(cfg, B, N, 1, workspace, workspace_bytes, true);
  if (st != RT_OK) return st;
  if (!layers || !emb || !ids || !k_caches || !v_caches || vocab <= 0 || N_max < N) return RT_ERR_INVALID_ARG;
  if (!aligned16(emb) || (hidden && !aligned16(hidden)) || (g_final && !aligned16(g_final))) return RT_ERR_INVALID_ARG;
  for (int l = 0; l < n_layers; ++l) {
    if (!weights_ok(&layers[l]) || !k_caches[l] || !v_caches[l] || !aligned16(k_caches[l]) || !aligned16(v_caches[l]))
      return RT_ERR_INVALID_ARG;
  }
  if ((size_t)B * cfg->d_model * 4 > 200 * 1024) return RT_ERR_UNSUPPORTED;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  unsigned char* ws = (unsigned char*)workspace;
  WsLayout L = ws_layout(cfg, B, N, n_layers);
  if (workspace_bytes < L.total)                               // what there is beyond a single layer's goes to layers side by side
    L = ws_layout(cfg, B, N, 1, (workspace_bytes - ws_layout(cfg, B, N, 1).total) & ~(size_t)255);
  if (cudaMemsetAsync(ws + L.sync, 0, sizeof(SyncArea), s) != cudaSuccess) return RT_ERR_CUDA;
  if (cudaMemsetAsync(ws + L.ll, 0, L.ll_bytes, s) != cudaSuccess) return RT_ERR_CUDA;
  const long long d = cfg->d_model;
  void* bufs[2] = {ws + L.hid0, ws + L.hid1};
  CallCtx ctx{s};
  {
    ProfScope ps(s, kProfOther);
    if (embed_launch(cfg->dtype, emb, ids, B, N, (int)d, vocab, bufs[0], s) != cudaSuccess) return RT_ERR_CUDA;
  }
  const void* cur = bufs[0];
  Wave wv = stack_wave(cfg, B, N, n_layers, L.form_bytes);
  if (wv.places && caches_overlap(cfg, n_layers, B, N, k_caches, v_caches)) wv.places = 0;
  ctx.exact = wv.exact != 0;
  if (wv.places) {
    st = run_stack_wave(cfg, n_layers, layers, bufs, hidden, B, N, k_caches, v_caches, N_max, ws, L, wv, ctx);
    if (st != RT_OK) return st;
    cur = hidden ? hidden : bufs[n_layers & 1];
  }
  for (int l = 0; l < n_layers && !wv.places; ++l) {
    void* out = (l == n_layers - 1 && hidden) ? hidden : bufs[(l + 1) & 1];
    st = run_layer(cfg, &layers[l], cur, (long long)N * d, d, out, (long long)N * d, d, B, N, 0, k_caches[l],
                   v_caches[l], N_max, ws, L, ctx);
    if (st != RT_OK) return st;
    cur = out;
  }
  if (logits_last) {
    ProfScope ps(s, kProfOther);
    const unsigned char* last = (const unsigned char*)cur + (size_t)(N - 1) * d * esize_of(cfg->dtype);
    if (head_launch(cfg->dtype, emb, g_final, last, (long long)N * d, B, (int)d, vocab, cfg->norm_flags, cfg->rms_eps,
                    logits_last, s) != cudaSuccess)
      return RT_ERR_CUDA;
  }
  return RT_OK;
}

rt_status rt_decode_step(const rt_config* cfg, int32_t n_layers, const rt_layer_weights* layers, const void* emb,
                         const void* g_final, int32_t vocab, const int32_t* ids, int32_t B, int32_t pos, float* logits,
                         void* const* k_caches, void* const* v_caches, int32_t N_max, void* workspace,
                         size_t workspace_bytes, void* cuda_stream) {
  rt_status st = common_checks(cfg, B, 1, n_layers, workspace, workspace_bytes);
  if (st != RT_OK) return st;
  if (!layers || !emb || !ids || !logits || !k_caches || !v_caches || vocab <= 0 || pos < 0 || pos >= N_max)
    return RT_ERR_INVALID_ARG;
  if (!aligned16(emb) || (g_final && !aligned16(g_final))) return RT_ERR_INVALID_ARG;
  for (int l = 0; l < n_layers; ++l) {
    if (!weights_ok(&layers[l]) || !k_caches[l] || !v_caches[l] || !aligned16(k_caches[l]) || !aligned16(v_caches[l]))
      return RT_ERR_INVALID_ARG;
  }
  if ((size_t)B * cfg->d_model * 4 > 200 * 1024) return RT_ERR_UNSUPPORTED;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  unsigned char* ws = (unsigned char*)workspace;
  const WsLayout L = ws_layout(cfg, B, 1, n_layers);
  if (cudaMemsetAsync(ws + L.sync, 0, sizeof(SyncArea), s) != cudaSuccess) return RT_ERR_CUDA;
  const long long d = cfg->d_model;
  rt_config c = *cfg;
  c.sched = RT_SCHED_NAIVE;
  void* bufs[2] = {ws + L.hid0, ws + L.hid1};
  if (decode_fast(cfg, B)) {
    // the last launch's output goes to the buffer that the last but one does not use
    void* z = bufs[(ceil_div(n_layers, kDecMaxLayers) - 1) & 1];
    st = run_decode(cfg, n_layers, layers, nullptr, 0, emb, ids, vocab, B, pos, z, d, k_caches, v_caches, ws, L, bufs, emb,
                    (size_t)vocab * d * 2, s);
    if (st != RT_OK) return st;
    return head_launch(c.dtype, emb, g_final, z, d, B, (int)d, vocab, c.norm_flags, c.rms_eps, logits, s) == cudaSuccess ? RT_OK : RT_ERR_CUDA;
  }
  if (cudaMemsetAsync(ws + L.ll, 0, L.ll_bytes, s) != cudaSuccess) return RT_ERR_CUDA;
  CallCtx ctx{s};
  if (embed_launch(c.dtype, emb, ids, B, 1, (int)d, vocab, bufs[0], s) != cudaSuccess) return RT_ERR_CUDA;
  const void* cur = bufs[0];
  for (int l = 0; l < n_layers; ++l) {
    void* out = bufs[(l + 1) & 1];
    st = run_layer(&c, &layers[l], cur, d, d, out, d, d, B, 1, pos, k_caches[l], v_caches[l], N_max, ws, L, ctx);
    if (st != RT_OK) return st;
    cur = out;
  }
  if (head_launch(c.dtype, emb, g_final, cur, d, B, (int)d, vocab, c.norm_flags, c.rms_eps, logits, s) != cudaSuccess)
    return RT_ERR_CUDA;
  return RT_OK;
}

rt_status rt_get_status(const void* workspace) {
  if (!workspace) return RT_ERR_INVALID_ARG;
  int st = 0;
  if (cudaMemcpy(&st, workspace, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return RT_ERR_CUDA;
  return (rt_status)st;
}

rt_status rt_update_tile(const rt_config* cfg, const void* q, const void* k_cache, const void* v_cache, float* st_o,
                         float* st_m, float* st_l, int32_t B, int32_t rows_q, int32_t rows_kv, int32_t q0, int32_t q1,
                         int32_t k0, int32_t k1, const float* alibi_slopes, void* workspace, void* cuda_stream) {
  if (!config_ok(cfg) || B <= 0 || !q || !k_cache || !v_cache || !st_o || !st_m || !st_l || !workspace)
    return RT_ERR_INVALID_ARG;
  if (q0 < 0 || q1 < q0 || q1 > rows_q || k0 < 0 || k1 < k0 || k1 > rows_kv) return RT_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k_cache) || !aligned16(v_cache) || !aligned16(st_o) || !aligned16(workspace))
    return RT_ERR_INVALID_ARG;
  const rt_status sup = config_supported(cfg, B, true);        // a tile takes any batch
  if (sup != RT_OK) return sup;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  if (cudaMemsetAsync(workspace, 0, sizeof(SyncArea), s) != cudaSuccess) return RT_ERR_CUDA;
  TileParams tp;
  memset(&tp, 0, sizeof(tp));
  tp.B = B; tp.d = cfg->d_model; tp.H = cfg->n_heads; tp.scale_log2 = cfg->softmax_scale * kLog2e; tp.alibi = alibi_slopes;
  tp.q = q; tp.k_cache = k_cache; tp.v_cache = v_cache;
  tp.st_o = st_o; tp.st_m = st_m; tp.st_l = st_l;
  tp.q0 = q0; tp.q1 = q1; tp.k0 = k0; tp.k1 = k1;
  tp.rows_q = rows_q; tp.rows_kv = rows_kv; tp.sync = (SyncArea*)workspace;
  ProfScope ps(s, kProfTile);
  return tile_launch(cfg->dtype, tp, s) == cudaSuccess ? RT_OK : RT_ERR_CUDA;
}

rt_status rt_selftest_wait_expiry(void* workspace, void* cuda_stream) {
  if (!workspace || !aligned16(workspace)) return RT_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  if (cudaMemsetAsync(workspace, 0, sizeof(SyncArea), s) != cudaSuccess) return RT_ERR_CUDA;
  return wait_expiry_selftest_launch((SyncArea*)workspace, s) == cudaSuccess ? RT_OK : RT_ERR_CUDA;
}

rt_status rt_profile_enable(int32_t on) {
  std::lock_guard<std::mutex> g(g_prof_mu);
  g_prof_on = on != 0;
  g_prof_timers = on >= 2;
  return RT_OK;
}

rt_status rt_profile_read(rt_profile* out) {
  if (!out) return RT_ERR_INVALID_ARG;
  memset(out, 0, sizeof(*out));
  std::vector<ProfSpan> spans;
  {
    std::lock_guard<std::mutex> g(g_prof_mu);
    spans.swap(g_prof_spans);
  }
  rt_status st = RT_OK;
  for (const ProfSpan& sp : spans) {
    float ms = 0.f;
    if (cudaEventSynchronize(sp.b) != cudaSuccess || cudaEventElapsedTime(&ms, sp.a, sp.b) != cudaSuccess) st = RT_ERR_CUDA;
    else { out->ms[sp.cls] += ms; out->launches[sp.cls] += 1; }
    cudaEventDestroy(sp.a);
    cudaEventDestroy(sp.b);
  }
  return st;
}

const char* rt_status_string(rt_status s) {
  switch (s) {
    case RT_OK: return "ok";
    case RT_ERR_INVALID_ARG: return "invalid argument";
    case RT_ERR_UNSUPPORTED: return "unsupported configuration";
    case RT_ERR_WORKSPACE: return "workspace too small";
    case RT_ERR_CUDA: return "CUDA runtime error";
    case RT_ERR_TIMEOUT: return "device-side wait timed out";
  }
  return "unknown status";
}

int32_t rt_plan_tiles(int32_t N, int32_t leaf, int32_t* out, int32_t cap) {
  if (N <= 0 || leaf <= 0) return 0;
  int32_t n = 0;
  for (int s0 = 0; s0 < N; s0 += leaf) {
    const int e0 = s0 + leaf < N ? s0 + leaf : N;
    if (e0 >= N) break;
    const int blocks = e0 / leaf;
    const int P = leaf * (blocks & -blocks);
    if (out && n < cap) {
      out[4 * n + 0] = e0; out[4 * n + 1] = e0 + P < N ? e0 + P : N;
      out[4 * n + 2] = e0 - P; out[4 * n + 3] = e0;
    }
    ++n;
  }
  return n;
}

rt_status rt_plan_counters(const rt_config* cfg, int32_t B, int32_t N, int32_t n_layers, int32_t vocab,
                           rt_counters* out) {
  if (!config_ok(cfg) || B <= 0 || N <= 0 || n_layers <= 0 || vocab < 0 || !out) return RT_ERR_INVALID_ARG;
  memset(out, 0, sizeof(*out));
  const uint64_t e = esize_of(cfg->dtype), d = cfg->d_model, H = cfg->n_heads, f = cfg->d_ff, b = B, n = N;
  const uint64_t tok = b * n;
  uint64_t rd = 0, wr = 0, kv = 0, kv_leaf = 0, fl_tile = 0, fl_leaf = 0, tiles = 0, leaves = 0;
  // pre-pass: RMS (x -> n), projection (n, W -> q, k~, v~), state seed (q, k~, v~ -> o, m, l)
  rd += tok * d * e + tok * d * e + 3 * d * d * e + 3 * tok * d * e;
  wr += tok * d * e + 3 * tok * d * e + tok * d * 4 + 2 * tok * H * 4;
  const uint64_t chain_w = (3 * d * d + 2 * d * f) * e;
  // per token: q row, carried state, x row in; z, k, v rows out
  rd += tok * d * e + tok * (d + 2 * H) * 4 + tok * d * e;
  wr += 3 * tok * d * e;
  fl_leaf += tok * 2 * (3 * d * d + 2 * d * f);
  if (cfg->sched == RT_SCHED_NAIVE) {
    leaves = 1;
    rd += chain_w;
    kv = b * d * e * n * (n - 1);                        // K and V rows of the whole prefix, every position
    fl_leaf += 4 * d * b * (n * (n - 1) / 2);
  } else {
    // the schedule that runs: leaf (or block) granularity of the chain form this shape takes
    const Schedule plan = effective_schedule(cfg, B, N);
    const Wave wv = stack_wave(cfg, B, N, n_layers, SIZE_MAX);             // layers side by side: every leaf meets all earlier pairs at once
    const uint64_t Lf = wv.places ? wv.leaf : plan.leaf;
    for (uint64_t s0 = 0; s0 < n; s0 += Lf) {
      const uint64_t e0 = s0 + Lf < n ? s0 + Lf : n, len = e0 - s0;
      ++leaves;
      // persistent kernels stage their weight rows once per leaf launch; dense products (wide batches, block sweeps)
      // stream them once per position resp. once per block (the group kernel re-reads them from L2)
      rd += chain_w * (plan.path == kPathWide ? len : (plan.path == kPathMmaSplit || plan.path == kPathGroups ? (b + plan.sub - 1) / plan.sub : 1));
      kv_leaf += 2 * b * d * e * (len * (len - 1) / 2);  // in-leaf pairs: written a few steps earlier, L2-resident
      fl_leaf += 4 * d * b * (len * (len - 1) / 2);
      if (e0 < n) {
        const uint64_t blocks = e0 / Lf;
        const uint64_t P = wv.places ? e0 : Lf * (blocks & (~blocks + 1));
        const uint64_t nq = (wv.places ? (e0 + Lf < n ? e0 + Lf : n) : (e0 + P < n ? e0 + P : n)) - e0;
        ++tiles;
        kv += 2 * P * b * d * e;
        rd += nq * b * d * e + nq * b * (d + 2 * H) * 4;
        wr += nq * b * (d + 2 * H) * 4;
        fl_tile += 4 * nq * P * d * b;
      }
    }
  }
  rd += kv;
  out->model_bytes_read = rd * n_layers;
  out->model_bytes_written = wr * n_layers;
  out->kv_bytes_read = kv * n_layers;
  out->leaf_kv_bytes_l2 = kv_leaf * n_layers;
  out->flops_tile = fl_tile * n_layers;
  out->flops_leaf = fl_leaf * n_layers;
  out->flops_gemm = tok * 2 * d * 3 * d * n_layers;
  out->n_tiles = tiles * n_layers;
  out->n_leaves = leaves * n_layers;
  if (vocab > 0) {
    out->model_bytes_read += tok * d * e + (uint64_t)vocab * d * e;
    out->model_bytes_written += tok * d * e + b * (uint64_t)vocab * 4;
    out->flops_gemm += 2 * b * d * (uint64_t)vocab;
  }
  return RT_OK;
}

}  // extern "C"
