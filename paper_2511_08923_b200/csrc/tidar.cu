// C-ABI entry points and per-step orchestration of the TiDAR decode path.
#include "../../include/tidar.h"

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <string>
#include <deque>
#include <vector>

#include "common.cuh"
#include "kernels_basic.cuh"
#include "kernels_replay.cuh"
#include "gemm_tc.cuh"
#include "attn_tc.cuh"

namespace {

constexpr int NORM_SMEM = 200 * 1024;  // shared memory of an SM that the norm kernel's blocks may claim between them
constexpr int MAX_SMS = 160;      // scratch is sized for this many (a B200 has 148)

std::string g_init_error;

struct SeqState {
  int n = 0;            // committed KV length
  int k = 0;            // draft block length of the sequence's last pass (entries its block holds)
  bool active = false;
  std::vector<int> pages;
};

struct TimedLaunch { int cls; cudaEvent_t a, b; };

}  // namespace

struct tidar_ctx {
  tidar_config cfg;
  cudaStream_t stream = nullptr;
  // borrowed weights
  const bf16 *embed = nullptr, *lm_head = nullptr, *final_norm = nullptr;
  std::vector<const bf16 *> attn_norm, wqkv, wo, ffn_norm, wgu, wdown;
  std::vector<const bf16 *> bqkv, q_norm, k_norm;      // optional (empty = absent)
  // geometry
  int R_head = 0;                  // rows of a pass that can get logits (the rows of a decode step)
  int head_row0 = 0;               // first row of the current pass that the LM head runs on
  int last_hidden_off = 0;         // first row of the last pass that the read-back calls address
  int R_cap = 0, T_max = 0, pages_per_seq = 0, n_pages = 0, n_qkv = 0, S_max = 4, lm_chunk = 0;
  size_t pool_stride = 0;    // elements in one layer's K (or V) pool
  size_t partial_stride = 0; // elements between split-K partial slabs
  size_t partials_cap = 0;   // floats in `partials`
  // arena carve-out (device)
  bf16 *kv = nullptr;
  RowMeta meta{};
  int32_t *d_blk_len = nullptr;    // [max_batch]: drafts a sequence's block holds (the block length of its last pass)
  // a step whose sequences use different block lengths: per listed sequence its k, first row, first local row;
  // per attention unit (two query tiles) its first row and the end of its sequence's rows
  int32_t *d_step_k = nullptr, *d_step_off = nullptr, *d_step_loc = nullptr, *d_unit_row0 = nullptr, *d_unit_rend = nullptr;
  int32_t *h_lay = nullptr;        // pinned staging for those five arrays
  size_t lay_ints = 0;
  int mixed_units = 0;             // attention units of the current mixed step
  float *d_run_max = nullptr, *d_run_sum = nullptr, *d_tgt_logit = nullptr, *d_logprob = nullptr;   // likelihood scoring, per row
  int32_t *d_target = nullptr;
  struct WMap { CUtensorMap full, small; };   // a weight matrix for the full and the SMALL instances of the projection kernel
  int32_t *d_seq_len = nullptr, *d_block = nullptr, *d_page_table = nullptr, *d_step_seqs = nullptr, *d_forced = nullptr,
          *d_step_n = nullptr, *d_step_L = nullptr, *d_prompt = nullptr, *d_arg_idx = nullptr;
  float *X = nullptr, *partials = nullptr, *rope_cos = nullptr, *rope_sin = nullptr, *d_arg_val = nullptr,
        *dbg_hidden = nullptr, *dbg_logits = nullptr;
  bf16 *A = nullptr, *Q = nullptr, *Kloc = nullptr, *Vloc = nullptr, *O = nullptr, *H = nullptr, *dbg_kv = nullptr;
  // host state
  std::vector<SeqState> seqs;
  std::vector<int> step_n;         // lengths of the sequences of the step being enqueued
  std::vector<int> free_pages;
  int32_t *h_pinned = nullptr;     // [max_batch*(k_max+1)] results + staging
  std::string err;
  int64_t launches = 0;
  // last pass
  int last_rows = 0, last_first_pos = 0;
  // Steps that have been enqueued and not yet waited for, oldest first.  Two may be in flight when every
  // acceptance length is forced (the host then knows the lengths without reading the device): the second
  // is enqueued while the first runs, so the device never waits for the host between steps.
  struct Flight { std::vector<int> seqs, ks; int k = 0, turn = 0; bool counted = false; };
  std::deque<Flight> inflight;
  cudaEvent_t flight_done[2] = {nullptr, nullptr};  // recorded behind the kernels of a slot's step
  int32_t *h_out2[2] = {nullptr, nullptr}, *h_stage2[2] = {nullptr, nullptr}, *h_done2[2] = {nullptr, nullptr};     // pinned, one set per slot (see StepIo)
  int32_t *h_page_table = nullptr;   // pinned mirror of the page table: the source of its (asynchronous) updates
  int turn = 0;                      // steps enqueued so far; step i uses slot i & 1
  // tensor-core path
  gemm_tc::EncodeTiledFn encode = nullptr;
  std::vector<WMap> tm_wqkv, tm_wo, tm_wgu, tm_wdown;
  WMap tm_lm;
  struct AMap { const void *p; int rows, cols, box; bool small; CUtensorMap tm; };
  std::vector<AMap> amaps;
  CUtensorMap tm_q, tm_kv, tm_kloc, tm_vloc;
  float *attn_part_O = nullptr; float2 *attn_part_ml = nullptr;
  attn_tc::Item *plan_items = nullptr; attn_tc::Tile *plan_tiles = nullptr;       // attention work plan of the current pass
  int n_sms = 0;
  // the launches of one decode step as an executable graph, valid for one key; the most recently used ones are kept
  struct StepKey {
    int k = 0, n_seqs = 0, mixed_R = 0, units = 0, mixed_K = 0; bool ar = false, timeline = false, count_tiles = false, split = false; int cluster = 1;
    bool operator==(const StepKey &o) const {
      return k == o.k && n_seqs == o.n_seqs && mixed_R == o.mixed_R && units == o.units && mixed_K == o.mixed_K && ar == o.ar && timeline == o.timeline &&
             count_tiles == o.count_tiles && split == o.split && cluster == o.cluster;
    }
  };
  struct StepGraph { StepKey key; cudaGraphExec_t exec = nullptr; int64_t launches = 0; std::vector<int> tl_cls; };   // tl_cls: of its timeline slots
  static constexpr size_t MAX_GRAPHS = 16;
  std::deque<StepGraph> graphs;      // most recently used first
  bool split_keys = true;            // attention key ranges of the current pass may be cut (see attention_plan)
  int attn_cluster = 1;              // CTAs that share an attention item of the current pass (see step_attention)
  struct { int cluster = 1; bool merge = false; int plan_units = 0; } route;     // of the last step or stand-alone attention (tidar_debug_attention_route)
  int max_clusters[attn_tc::MAX_CLUSTER + 1] = {};      // clusters of 2, 4, 8 attention CTAs that are resident at once
  bool graphs_ok = true;             // steps can be captured on this stream (the legacy default stream refuses it)
  // On the legacy default stream a step is captured on a stream of the context's own, once its shape has been run GRAPH_AFTER times, and replayed
  // on the default stream from then on (see launch_step).
  bool side_capture = false;
  cudaStream_t capture_stream = nullptr;
  std::deque<std::pair<StepKey, int>> seen;      // shapes without a graph and how often they were run, most recent first
  int64_t graphs_captured = 0, graphs_launched = 0;
  bool slab_bf16 = false;          // split-K partial sums of the step in bf16 instead of fp32 (config debug bit 2)
  int32_t *d_status = nullptr, *cand_idx = nullptr;
  float *cand_val = nullptr;
  // in-kernel timeline (diagnostics): two words per launch of the last recorded step
  static constexpr int TL_MAX = 2048;
  unsigned long long *d_tl = nullptr;
  bool timeline = false; int tl_n = 0; std::vector<int> tl_cls;
  bool count_tiles = false;        // the attention kernel adds the key tiles it visits to d_tl[2 * TL_MAX]
  float tl_class_ms[TIDAR_TC_COUNT] = {}; float tl_span_ms = 0.f, tl_busy_ms = 0.f;
  // timing
  bool timing = false; std::vector<TimedLaunch> timed; float class_ms[TIDAR_TC_COUNT] = {};
  int cur_class = 0;
};

namespace {

int fail(tidar_ctx *c, int code, const char *fmt, ...) {
  char buf[512];
  va_list ap; va_start(ap, fmt); vsnprintf(buf, sizeof buf, fmt, ap); va_end(ap);
  if (c) c->err = buf; else g_init_error = buf;
  return code;
}

#define CUDA_TRY(c, call)                                                                     \
  do {                                                                                        \
    cudaError_t e_ = (call);                                                                  \
    if (e_ != cudaSuccess) return fail((c), TIDAR_ECUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
  } while (0)

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Lays the arena out; with base == nullptr only measures.
struct Carver {
  char *base; size_t off = 0;
  explicit Carver(void *b) : base((char *)b) {}
  template <typename T> T *take(size_t n) {
    off = align_up(off, 256);
    T *p = base ? (T *)(base + off) : nullptr;
    off += n * sizeof(T);
    return p;
  }
};

int validate(const tidar_config &c, std::string &why) {
  auto bad = [&](const char *m) { why = m; return TIDAR_EINVAL; };
  if (c.n_layers < 1 || c.d_model < 64 || c.vocab < 2 || c.d_ffn < 64) return bad("n_layers, d_model, d_ffn, vocab must be positive");
  if (c.head_dim != 64 && c.head_dim != 128) return bad("head_dim must be 64 or 128");
  if (c.n_kv_heads < 1 || c.n_q_heads < 1 || c.n_q_heads % c.n_kv_heads) return bad("n_q_heads must be a positive multiple of n_kv_heads");
  if (c.n_q_heads / c.n_kv_heads > 128) return bad("at most 128 query heads per KV head (one 128-row attention tile)");
  if (c.d_model > 12288) return bad("d_model above 12288 is not supported (row buffer of the norm kernel)");
  if (c.d_model % 64 || c.d_ffn % 64) return bad("d_model and d_ffn must be multiples of 64");
  if (c.page_size != 64) return bad("page_size must be 64");
  if (c.k_max < 1 || c.k_max > 32) return bad("k_max must be in [1, 32]");
  if (c.max_batch < 1 || c.max_seq_len < 2 * c.k_max + 1) return bad("max_batch >= 1 and max_seq_len > 2*k_max required");
  if (c.mask_token_id < 0 || c.mask_token_id >= c.vocab) return bad("mask_token_id out of range");
  if (!(c.beta >= 0.0f && c.beta <= 1.0f)) return bad("beta must be in [0, 1]");
  if (!(c.temperature >= 0.0f) || c.temperature > 1e4f) return bad("temperature must be in [0, 1e4] (0 = greedy)");
  if (c.impl != 0 && c.impl != 1) return bad("impl must be 0 (tensor-core kernels) or 1 (replay kernels)");
  if (c.prefill_rows < 0 || c.prefill_rows > (1 << 16)) return bad("prefill_rows must be in [0, 65536]");
  if (!(c.rms_eps > 0.f) || !(c.rope_theta > 1.f)) return bad("rms_eps > 0 and rope_theta > 1 required");
  return TIDAR_OK;
}

void layout(tidar_ctx &x, void *arena, size_t *bytes) {
  const tidar_config &c = x.cfg;
  x.T_max = c.k_max * (c.k_max + 1);
  // rows of a pass: the step's slots, plus one mixed row per verified position when beta < 1
  x.R_head = (int)align_up((size_t)std::max(c.max_batch * (x.T_max + (c.beta < 1.0f ? c.k_max : 0)), 256), 16);
  x.R_cap = std::max(x.R_head, (int)align_up((size_t)std::max(c.prefill_rows, 0), 16));
  x.pages_per_seq = (c.max_seq_len + c.page_size - 1) / c.page_size;
  x.n_pages = x.pages_per_seq * c.max_batch;
  x.n_qkv = (c.n_q_heads + 2 * c.n_kv_heads) * c.head_dim;
  x.pool_stride = (size_t)x.n_pages * c.n_kv_heads * c.page_size * c.head_dim;
  x.lm_chunk = std::min(c.vocab, 16384);
  x.S_max = c.impl == 0 ? MAX_SLABS : 4;
  const size_t R = x.R_cap;
  const size_t widest = std::max<size_t>({(size_t)x.S_max * x.n_qkv, (size_t)x.S_max * c.d_model, (size_t)2 * c.d_ffn,
                                          (size_t)x.lm_chunk, (size_t)2 * gemm_tc::lse_parts(c.vocab)});
  x.partial_stride = 0;  // set per projection
  Carver cv(arena);
  x.kv = cv.take<bf16>((size_t)c.n_layers * 2 * x.pool_stride);
  x.meta.ids = cv.take<int32_t>(R); x.meta.pos = cv.take<int32_t>(R); x.meta.seq = cv.take<int32_t>(R);
  x.meta.nvis = cv.take<int32_t>(R); x.meta.loc0 = cv.take<int32_t>(R); x.meta.nloc = cv.take<int32_t>(R);
  x.meta.cache_pos = cv.take<int32_t>(R); x.meta.local_idx = cv.take<int32_t>(R);
  x.meta.skey = cv.take<uint32_t>(R);
  x.d_seq_len = cv.take<int32_t>(c.max_batch);
  x.d_blk_len = cv.take<int32_t>(c.max_batch);
  // one block, so that one copy brings the whole layout of a mixed step over (same order in h_lay)
  x.lay_ints = 3 * (size_t)(c.max_batch + 1) + 2 * (size_t)(x.R_head + c.max_batch);
  x.d_step_k = cv.take<int32_t>(x.lay_ints);
  x.d_step_off = x.d_step_k + (c.max_batch + 1); x.d_step_loc = x.d_step_off + (c.max_batch + 1);
  x.d_unit_row0 = x.d_step_loc + (c.max_batch + 1); x.d_unit_rend = x.d_unit_row0 + (x.R_head + c.max_batch);
  x.d_run_max = cv.take<float>(R); x.d_run_sum = cv.take<float>(R); x.d_tgt_logit = cv.take<float>(R); x.d_logprob = cv.take<float>(R);
  x.d_target = cv.take<int32_t>(R);
  x.d_block = cv.take<int32_t>((size_t)c.max_batch * c.k_max);
  x.d_page_table = cv.take<int32_t>((size_t)c.max_batch * x.pages_per_seq);
  x.d_step_seqs = cv.take<int32_t>(c.max_batch); x.d_forced = cv.take<int32_t>(c.max_batch);
  x.d_step_n = cv.take<int32_t>(c.max_batch); x.d_step_L = cv.take<int32_t>(c.max_batch);
  x.d_prompt = cv.take<int32_t>(c.max_seq_len);
  x.d_arg_idx = cv.take<int32_t>(R); x.d_arg_val = cv.take<float>(R);
  x.d_status = cv.take<int32_t>(64);
  x.d_tl = cv.take<unsigned long long>(2 * tidar_ctx::TL_MAX + 8);   // timeline slots, then diagnostic counters
  if (c.impl == 0) {
    const size_t slots = (size_t)attn_tc::SLOTS_PER_SM * MAX_SMS;
    x.attn_part_O = cv.take<float>(slots * 2 * 128 * c.head_dim);
    x.attn_part_ml = cv.take<float2>(slots * 2 * 128);
    x.plan_tiles = cv.take<attn_tc::Tile>(2 * R);     // a unit of two query tiles holds at least one row
    x.plan_items = cv.take<attn_tc::Item>(std::max<size_t>(slots, R));
  }
  {
    const size_t G = 4 * 256;            // (CTAs of the LM-head kernel <= SMs) x 4 lane quadrants
    x.cand_val = cv.take<float>(G * R); x.cand_idx = cv.take<int32_t>(G * R);
  }
  x.X = cv.take<float>(R * c.d_model);
  x.partials = cv.take<float>(R * widest);
  x.partials_cap = R * widest;
  x.rope_cos = cv.take<float>(R * (c.head_dim / 2)); x.rope_sin = cv.take<float>(R * (c.head_dim / 2));
  x.A = cv.take<bf16>(R * c.d_model);
  x.Q = cv.take<bf16>(R * c.n_q_heads * c.head_dim);
  x.O = cv.take<bf16>(R * c.n_q_heads * c.head_dim);
  const size_t nloc = (size_t)std::max(c.max_batch * c.k_max * c.k_max, c.k_max);
  x.Kloc = cv.take<bf16>(nloc * c.n_kv_heads * c.head_dim);
  x.Vloc = cv.take<bf16>(nloc * c.n_kv_heads * c.head_dim);
  x.H = cv.take<bf16>(R * c.d_ffn);
  x.dbg_kv = cv.take<bf16>((size_t)2 * 256 * c.n_kv_heads * c.head_dim);
  if (c.debug & 1) {
    x.dbg_hidden = cv.take<float>((size_t)(c.n_layers + 1) * R * c.d_model);
    x.dbg_logits = cv.take<float>((size_t)x.R_head * (size_t)c.vocab);
  }
  *bytes = align_up(cv.off, 256);
}

// A kernel of a pass is launched with programmatic stream serialization: it may be scheduled while the previous
// kernel of the stream is still running and synchronises itself with pdl_wait(); only kernels that call
// pdl_wait() before they touch produced data may be launched this way.  Between a projection and the small kernel
// behind it (norm, RoPE) an ordinary dependency costs 2.3 - 4 us, this one 1.0 - 1.5.  What makes it pay is that the
// kernels fit beside one another: all ask for the same split of the SM's memory (an SM changes its split only when it is
// empty; see init_tensor_core_path).
template <typename... KP, typename... AP>
inline void launch_pdl_cluster(unsigned cluster, void (*kernel)(KP...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, AP &&...args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = cluster > 1 ? 2 : 1;
  cudaLaunchKernelEx(&cfg, kernel, KP(std::forward<AP>(args))...);
}
template <typename... KP, typename... AP>
inline void launch_pdl(void (*kernel)(KP...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, AP &&...args) {
  launch_pdl_cluster(1, kernel, grid, block, smem, st, std::forward<AP>(args)...);
}

// ---- launch bookkeeping -----------------------------------------------------
struct Launch {
  tidar_ctx *c; int cls; cudaEvent_t a = nullptr, b = nullptr; TlSlot tl{nullptr};
  Launch(tidar_ctx *c_, int cls_) : c(c_), cls(cls_) {
    c->launches++;
    if (c->timing) { cudaEventCreate(&a); cudaEventCreate(&b); cudaEventRecord(a, c->stream); }
    if (c->timeline && c->tl_n < tidar_ctx::TL_MAX) { tl.t = c->d_tl + 2 * c->tl_n; c->tl_n++; c->tl_cls.push_back(cls); }
  }
  ~Launch() {
    if (c->timing) { cudaEventRecord(b, c->stream); c->timed.push_back({cls, a, b}); }
  }
};

void collect_timing(tidar_ctx *c) {
  for (int i = 0; i < TIDAR_TC_COUNT; ++i) c->class_ms[i] = 0.f;
  for (auto &t : c->timed) {
    float ms = 0.f; cudaEventElapsedTime(&ms, t.a, t.b);
    c->class_ms[t.cls] += ms;
    cudaEventDestroy(t.a); cudaEventDestroy(t.b);
  }
  c->timed.clear();
}

// Per class, the sum over the last step's launches of (latest CTA end - earliest CTA start);
// busy = the sum over all launches, span = first start to last end.
void collect_timeline(tidar_ctx *c) {
  std::vector<unsigned long long> h(2 * (size_t)c->tl_n);
  for (int i = 0; i < TIDAR_TC_COUNT; ++i) c->tl_class_ms[i] = 0.f;
  c->tl_span_ms = c->tl_busy_ms = 0.f;
  if (c->tl_n == 0) return;
  if (cudaMemcpy(h.data(), c->d_tl, h.size() * sizeof(unsigned long long), cudaMemcpyDeviceToHost) != cudaSuccess) { cudaGetLastError(); return; }
  unsigned long long first = ~0ull, last = 0;
  for (int i = 0; i < c->tl_n; ++i) {
    if (h[2 * i] == 0 || h[2 * i + 1] == 0) continue;          // a launch that stamped nothing
    const unsigned long long t0 = ~h[2 * i], t1 = h[2 * i + 1];
    if (t1 < t0) continue;
    const float ms = (float)((double)(t1 - t0) * 1e-6);
    c->tl_class_ms[c->tl_cls[i]] += ms; c->tl_busy_ms += ms;
    first = std::min(first, t0); last = std::max(last, t1);
  }
  if (last > first) c->tl_span_ms = (float)((double)(last - first) * 1e-6);
}

KvGeom geom(const tidar_ctx *c) {
  return KvGeom{c->cfg.n_kv_heads, c->cfg.head_dim, c->cfg.page_size, c->pages_per_seq, c->d_page_table, 0};
}

// ---- projections --------------------------------------------------------------
bool encode_weights(tidar_ctx *c, tidar_ctx::WMap *tm, const void *p, int rows, int cols) {
  return gemm_tc::encode_2d(c->encode, &tm->full, p, (uint64_t)rows, (uint64_t)cols, gemm_tc::TILE_N) == CUDA_SUCCESS &&
         gemm_tc::encode_2d_small(c->encode, &tm->small, p, (uint64_t)rows, (uint64_t)cols, gemm_tc::TILE_N) == CUDA_SUCCESS;
}
// Tensor map of an activation matrix [rows][cols] (bf16) with a box of `box` rows; cached.
const CUtensorMap *act_map(tidar_ctx *c, const void *p, int rows, int cols, int box, bool small) {
  for (auto &m : c->amaps) if (m.p == p && m.rows == rows && m.cols == cols && m.box == box && m.small == small) return &m.tm;
  tidar_ctx::AMap m{p, rows, cols, box, small, {}};
  if ((small ? gemm_tc::encode_2d_small : gemm_tc::encode_2d)(c->encode, &m.tm, p, (uint64_t)rows, (uint64_t)cols, (uint32_t)box) != CUDA_SUCCESS) return nullptr;
  if (c->amaps.size() > 256) c->amaps.erase(c->amaps.begin());
  c->amaps.push_back(m);
  return &c->amaps.back().tm;
}

// CTAs of the LM head, each of which leaves four candidates per row (with several row blocks it may meet only some of the rows).
int lm_head_ctas(const tidar_ctx *c, int R, int vocab) {
  const int pairs = c->n_sms / 2, tiles = (vocab + gemm_tc::tile_rows(false) - 1) / gemm_tc::tile_rows(false);
  return 2 * (R <= gemm_tc::MAX_ROWS ? std::min(tiles, pairs) : pairs);
}
// Whether a projection runs as a SMALL instance (the LM head's argmax epilogue needs the registers of the full one).  Up to one
// block of SMALL_ROWS rows always.  Up to one block's worth of rows (MAX_ROWS), as several blocks of 96, where the weight
// matrix is small: such a launch is all start-up and slab store, both of which a SMALL CTA, which sits beside the kernels in
// front of it, hides better, and re-reading a few MB of weights per block from L2 costs less.  (1.5B-class step at 272 rows, its
// projections of 2.4 - 13.8 M weights: 2.18 -> 1.96 ms; 8B-class, from 16.8 M weights on: 1 % slower that way; the fused
// gate/up projection of 27.5 M weights: 12 % of the step slower.  15 M is simply a line between the two models measured: a matrix
// between 13.8 M and 16.8 M weights may do a per cent better on the other side.)
bool small_gemm(int mode, int R, int N, int K) {
  if (mode != gemm_tc::MODE_SLAB && mode != gemm_tc::MODE_SWIGLU) return false;
  return R <= gemm_tc::SMALL_ROWS || (mode == gemm_tc::MODE_SLAB && R <= gemm_tc::MAX_ROWS && (long long)N * K <= 15000000);
}

// Work of a tensor-core projection of R rows: row blocks, K splits, which tiles finish in the fused epilogue.
gemm_tc::Args plan_gemm(const tidar_ctx *c, int mode, int R, int N, int K, int force_S = 0) {
  gemm_tc::Args a{};
  a.R = R; a.N = N; a.K = K;
  const bool small = small_gemm(mode, R, N, K);
  const int max_rows = small ? gemm_tc::SMALL_ROWS : gemm_tc::MAX_ROWS;
  gemm_tc::plan_rows(R, a, (R + max_rows - 1) / max_rows);
  const int kps = gemm_tc::k_per_stage(small), tile = gemm_tc::tile_rows(small);
  const int workers = small ? c->n_sms : c->n_sms / 2;             // CTAs, or pairs of CTAs, that work on items
  a.n_tiles = (N + tile - 1) / tile;
  a.kb_total = (K / gemm_tc::TILE_K + kps - 1) / kps;
  a.S = 1; a.fused_items = 0; a.tile_b0 = 0; a.n_tiles_b = 0;
  const bool blocks = a.n_rb > 1 && !small;
  if (blocks) gemm_tc::plan_blocks(a, workers, mode == gemm_tc::MODE_SLAB ? c->S_max : 0, 4);
  if (mode == gemm_tc::MODE_SLAB) {
    a.n_tiles_b = a.n_tiles;
    a.S = force_S > 0 ? std::min(force_S, a.kb_total) : blocks ? a.S
                      : gemm_tc::plan_splits(a.n_rb * a.n_tiles, a.kb_total, workers, c->S_max, 4 / kps, 3.0 / kps);
    a.ldo = N; a.slab_stride = (long long)R * N;
  } else if (mode == gemm_tc::MODE_SWIGLU) {
    a.ldh = N / 2;
    a.fused_items = a.n_rb * a.n_tiles;
    // more tiles than SMs: whole waves of tiles finish in the fused epilogue; the tiles of the
    // last, partial wave are split along K so that they also fill the machine, and are finished
    // from fp32 slabs by swiglu_slab_kernel
    if (a.n_rb == 1 && a.n_tiles > workers && a.n_tiles % workers) {
      const int full = a.n_tiles / workers * workers;
      const int rem = a.n_tiles - full;
      const int S2 = std::min({workers / rem, a.kb_total * kps / 4, c->S_max});
      if (S2 >= 2 && (size_t)S2 * R * rem * tile <= c->partials_cap) {
        a.fused_items = full; a.tile_b0 = full; a.n_tiles_b = rem; a.S = S2;
        a.ldo = rem * tile; a.slab_stride = (long long)R * a.ldo;
      }
    }
  } else {
    a.fused_items = a.n_rb * a.n_tiles;
  }
  // Partial sums and additions to the residual stream are walked through ahead (see the kernel) where every worker has one item: its store is then the
  // end of the launch.  With more, the first item's store runs beside the second's main loop and fetches the code for the last, and a walk
  // only costs.  (Down projection of the 1.5B class, launches timed one by one: 1400 rows, 72 items on 74 workers, 37.3 us without and 35.7 with;
  // 1776 rows, 126 items, 45.7 and 47.6.)  And where the main loop, 2.15 cycles per row + 50 and K block at 1.75 GHz, is longer than the nap and the walk
  // leave behind: 16 K blocks of 272 rows and 24 of 160 gain, 12 of 208 (3.4 us) lose 0.3 us, 8 of 208 0.9, and a first pass of the tiny model, 4 and 11 K
  // blocks, 168 -> 176 us.
  const float loop_us = (float)((a.kb_total + a.S - 1) / a.S) * (2.15f * a.rb_rows + 50.f) / 1750.f;
  a.warm_epilogue = mode != gemm_tc::MODE_SLAB || (a.total_items() <= workers && loop_us >= 4.f);
  return a;
}

// Tensor-core projection.  A [a_rows][K] (first R rows used), W described by tmW ([N][K]).
//   MODE_SLAB  : S split-K partial slabs of fp32 [R][N] into c->partials (S chosen here); with `residual` [R][N] given and
//                nothing split, the result is added to it instead and *S_out is 0
//   MODE_SWIGLU: bf16 c->H [R][N/2]
//   MODE_ARGMAX: candidates for argmax_merge_kernel (+ optional logits dump)
//   MODE_LSE   : pieces of the rows' log-sum-exp in c->partials for score_merge_kernel, and the logits of `target` [R]
int gemm_tc_launch(tidar_ctx *c, int mode, const bf16 *A, int a_rows, const tidar_ctx::WMap &tmW, int R, int N, int K, int cls,
                   int *S_out, size_t *stride_out, float *slab_out = nullptr, int force_S = 0, float *residual = nullptr,
                   const int32_t *target = nullptr) {
  gemm_tc::Args a = plan_gemm(c, mode, R, N, K, force_S);
  const bool small = small_gemm(mode, R, N, K);
  const int rem_tiles = mode == gemm_tc::MODE_SWIGLU ? a.n_tiles_b : 0;
  if (mode == gemm_tc::MODE_SLAB) {
    a.out = slab_out ? (void *)slab_out : (void *)c->partials;
    a.slab_bf16 = (slab_out || !c->slab_bf16) ? 0 : 1;   // an explicit output buffer always gets exact fp32 slabs
    if (residual && a.S == 1 && !a.slab_bf16) { a.out = residual; a.accumulate = 1; }
  } else if (mode == gemm_tc::MODE_SWIGLU) {
    a.H = c->H;
    a.out = c->partials; a.slab_bf16 = c->slab_bf16 ? 1 : 0;
  } else if (mode == gemm_tc::MODE_LSE) {
    a.lse = reinterpret_cast<float2 *>(c->partials); a.target = target; a.tgt_logit = c->d_tgt_logit;
  } else {
    a.cand_val = c->cand_val; a.cand_idx = c->cand_idx; a.cand_ld = lm_head_ctas(c, R, N) * 4; a.dump = c->dbg_logits; a.ld_dump = c->cfg.vocab; a.col0 = 0;
    a.inv_temp = c->cfg.temperature > 0.f ? 1.0f / c->cfg.temperature : 0.f; a.skey = c->meta.skey + c->head_row0;
  }
  a.status = c->d_status;
  const int box = small ? a.rb_rows : a.rb_rows / 2;
  const CUtensorMap *tmA = act_map(c, A, a_rows, K, box, small);
  if (!tmA) return fail(c, TIDAR_ECUDA, "cuTensorMapEncodeTiled failed for an activation matrix (%d x %d, box %d)", a_rows, K, box);
  const int items = a.total_items();
  const int workers = std::min(items, small ? c->n_sms : c->n_sms / 2), grid = small ? workers : 2 * workers;
  {
    int n = 0;                                   // stages the first worker's items have
    for (int i = 0; i < items; i += workers) n += i < a.fused_items ? a.kb_total : (a.kb_total + a.S - 1) / a.S;
    gemm_tc::plan_stages(a, n, small);
  }
  const size_t smem = gemm_tc::smem_bytes(a, small);
  Launch l(c, cls);
  if (small && mode == gemm_tc::MODE_SLAB) launch_pdl(gemm_tc::gemm_tc_kernel<gemm_tc::MODE_SLAB, true>, grid, gemm_tc::THREADS, smem, c->stream, tmW.small, *tmA, a, l.tl);
  else if (small) launch_pdl(gemm_tc::gemm_tc_kernel<gemm_tc::MODE_SWIGLU, true>, grid, gemm_tc::THREADS, smem, c->stream, tmW.small, *tmA, a, l.tl);
  else if (mode == gemm_tc::MODE_SLAB) launch_pdl_cluster(2, gemm_tc::gemm_tc_kernel<gemm_tc::MODE_SLAB>, grid, gemm_tc::THREADS, smem, c->stream, tmW.full, *tmA, a, l.tl);
  else if (mode == gemm_tc::MODE_SWIGLU) launch_pdl_cluster(2, gemm_tc::gemm_tc_kernel<gemm_tc::MODE_SWIGLU>, grid, gemm_tc::THREADS, smem, c->stream, tmW.full, *tmA, a, l.tl);
  else if (mode == gemm_tc::MODE_LSE) launch_pdl_cluster(2, gemm_tc::gemm_tc_kernel<gemm_tc::MODE_LSE>, grid, gemm_tc::THREADS, smem, c->stream, tmW.full, *tmA, a, l.tl);
  else if (a.inv_temp > 0.f) launch_pdl_cluster(2, gemm_tc::gemm_tc_kernel<gemm_tc::MODE_SAMPLE>, grid, gemm_tc::THREADS, smem, c->stream, tmW.full, *tmA, a, l.tl);
  else launch_pdl_cluster(2, gemm_tc::gemm_tc_kernel<gemm_tc::MODE_ARGMAX>, grid, gemm_tc::THREADS, smem, c->stream, tmW.full, *tmA, a, l.tl);
  if (rem_tiles) {
    const int f0 = a.tile_b0 * gemm_tc::tile_rows(small) / 2, nf = N / 2 - f0;          // features of the split tiles
    const size_t n = (size_t)R * nf;
    Launch lf(c, cls);
    if (c->slab_bf16)
      launch_pdl(swiglu_slab_kernel<bf16>, (unsigned)((n / 2 + 255) / 256), 256, 0, c->stream, (const bf16 *)c->partials, a.S, (size_t)a.slab_stride, R, a.ldo, nf,
                                                                           f0, a.ldh, c->H, lf.tl);
    else
      launch_pdl(swiglu_slab_kernel<float>, (unsigned)((n / 2 + 255) / 256), 256, 0, c->stream, (const float *)c->partials, a.S, (size_t)a.slab_stride, R, a.ldo, nf,
                                                                           f0, a.ldh, c->H, lf.tl);
  }
  if (S_out) *S_out = a.accumulate ? 0 : a.S;
  if (stride_out) *stride_out = (size_t)R * N;
  return TIDAR_OK;
}

enum Proj { P_QKV, P_O, P_GU, P_DOWN };

// out = A[R][K] * W[N][K]^T as S split-K partial slabs of fp32 [R][N] (replay: S = 1).
int gemm_partials(tidar_ctx *c, const bf16 *A, int a_rows, const bf16 *W, const tidar_ctx::WMap *tmW, int R, int N, int K, float *out,
                  int *S_out, size_t *stride_out, int cls, float *residual = nullptr) {
  if (c->cfg.impl == 0) return gemm_tc_launch(c, gemm_tc::MODE_SLAB, A, a_rows, *tmW, R, N, K, cls, S_out, stride_out, nullptr, 0, residual);
  Launch l(c, cls);
  dim3 grid((N + 63) / 64, (R + 63) / 64);
  gemm_replay_kernel<<<grid, 256, 0, c->stream>>>(A, K, W, K, out, N, R, N, K);
  *S_out = 1; *stride_out = (size_t)R * N;
  return TIDAR_OK;
}

// bf16 tensor maps for the attention kernel (128-byte swizzle, 64-element inner box).
bool encode_q_map(tidar_ctx *c, CUtensorMap *tm, const void *q, int rows) {
  const tidar_config &cf = c->cfg;
  const int G = cf.n_q_heads / cf.n_kv_heads, spt = 128 / G;
  cuuint64_t dims[3] = {(cuuint64_t)cf.head_dim, (cuuint64_t)cf.n_q_heads, (cuuint64_t)rows};
  cuuint64_t strides[2] = {(cuuint64_t)cf.head_dim * 2, (cuuint64_t)cf.n_q_heads * cf.head_dim * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)G, (cuuint32_t)spt}, es[3] = {1, 1, 1};
  return c->encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(q), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// K or V pages [page][kv head][64][head_dim]; a load brings one page of one KV head, the 64-element halves of the head one behind the other.
bool encode_pages_map(tidar_ctx *c, CUtensorMap *tm, const void *pool, long long n_pages) {
  const tidar_config &cf = c->cfg;
  const cuuint64_t row = (cuuint64_t)cf.head_dim * 2;
  cuuint64_t dims[5] = {64, 64, (cuuint64_t)cf.head_dim / 64, (cuuint64_t)cf.n_kv_heads, (cuuint64_t)n_pages};
  cuuint64_t strides[4] = {row, 128, 64 * row, (cuuint64_t)cf.n_kv_heads * 64 * row};
  cuuint32_t box[5] = {64, 64, (cuuint32_t)cf.head_dim / 64, 1, 1}, es[5] = {1, 1, 1, 1, 1};
  return c->encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(pool), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// Step-local K or V rows [row][kv head][head_dim]; a load brings 64 rows in the layout of a page.
bool encode_local_map(tidar_ctx *c, CUtensorMap *tm, const void *loc, long long rows) {
  const tidar_config &cf = c->cfg;
  const cuuint64_t head = (cuuint64_t)cf.head_dim * 2;
  cuuint64_t dims[4] = {64, (cuuint64_t)rows, (cuuint64_t)cf.head_dim / 64, (cuuint64_t)cf.n_kv_heads};
  cuuint64_t strides[3] = {(cuuint64_t)cf.n_kv_heads * head, 128, head};
  cuuint32_t box[4] = {64, 64, (cuuint32_t)cf.head_dim / 64, 1}, es[4] = {1, 1, 1, 1};
  return c->encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(loc), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct AttnMaps { const CUtensorMap *q, *k, *v, *kloc, *vloc; int page_base_k, page_base_v; };

// Units (up to two query tiles of one sequence) of a pass of R rows.  rows_per_group: slots per sequence (k(k+1) in a
// step; all rows in a first-pass chunk); <= 0: the sequences' groups differ in size and the units come from the mixed
// step's table.  Key ranges may be split (see attn_tc::plan_block) while there are fewer than three
// (unit, KV head) combinations for two SMs: beyond that they fill the machine evenly enough.
// c->split_keys == false: no key range of the pass is long enough to be worth cutting (see may_split).
// The grid is the number of items the plan may use; a CTA holds a whole SM, so up to one combination per SM it is one wave.
attn_tc::PlanArgs attention_plan(const tidar_ctx *c, int R, int rows_per_group) {
  const tidar_config &cf = c->cfg;
  attn_tc::PlanArgs p{};
  p.R = R; p.spt = 128 / (cf.n_q_heads / cf.n_kv_heads); p.Hkv = cf.n_kv_heads;
  if (rows_per_group > 0) {
    p.rows_per_group = rows_per_group;
    p.units_per_group = (rows_per_group + 2 * p.spt - 1) / (2 * p.spt);
    p.n_units = (R + rows_per_group - 1) / rows_per_group * p.units_per_group;
  } else {
    p.rows_per_group = R; p.units_per_group = 1;
    p.unit_row0 = c->d_unit_row0; p.unit_rend = c->d_unit_rend; p.n_units = c->mixed_units;
  }
  p.n_sms = c->n_sms;
  const int units = p.n_units * p.Hkv;
  static_assert(attn_tc::PLAN_UNITS >= 3 * MAX_SMS / 2, "units that may be split are planned");
  p.max_items = units <= c->n_sms ? c->n_sms / p.Hkv : 2 * units < 3 * c->n_sms ? attn_tc::SLOTS_PER_SM * c->n_sms / p.Hkv : p.n_units;
  p.max_pieces = attn_tc::MAX_SPLITS;
  if (!c->split_keys) { p.max_pieces = 1; p.max_items = 2 * units <= c->n_sms ? 2 * p.n_units : p.n_units; }
  if (c->attn_cluster > 1) {                           // one item per tile, shared by a cluster
    p.max_pieces = 1; p.singles = 1;
    p.max_items = rows_per_group > 0 ? (R + rows_per_group - 1) / rows_per_group * ((rows_per_group + p.spt - 1) / p.spt) : 2 * p.n_units;
  }
  p.items = c->plan_items; p.tiles = c->plan_tiles;
  return p;
}

// Whether a pass whose rows see at most n_keys positions may cut key ranges.  A cut costs a partial result's store and the merge
// kernel, about 5 us, and saves half of 0.56 us per page at best.
bool may_split(int n_keys) { return n_keys > 12 * attn_tc::PAGE; }

// The same for a decode step, whose sequences' lengths n[] and block lengths (ks[], or k for all) the host knows: whether the work plan
// (attn_tc::plan_block, from the same estimate) would cut any key range.  Where it would not, the step goes without the merge kernel, which would find nothing
// to do (8B-class step of 272 rows, 1.1 k positions: 2.4 us per layer).  A step planned as uncut on the host is not cut on the device.
// This runs ahead of every step's first launch, so equal units are counted and not listed, nothing is allocated, and a block length's tiles are worked
// out once for all sequences next to one another that have it (12/2 heads, 60 sequences of one row: 11.3 -> 2.8 us; 14 of 272 rows: 22.5 -> 5.1).
struct StepAttention { bool split; int cluster; };
StepAttention step_attention(const tidar_ctx *c, const int *n, const int *ks, int k_all, int n_seqs, bool ar, bool mixed) {
  using namespace attn_tc;
  const StepAttention uncut{false, 1}, cut{true, 1};
  const int spt = 128 / (c->cfg.n_q_heads / c->cfg.n_kv_heads), Hkv = c->cfg.n_kv_heads;
  auto rows = [&](int s) { const int k = ks ? ks[s] : k_all; return ar ? 1 : k * (k + 1); };
  int n_units = 0, longest = 0;
  for (int s = 0; s < n_seqs; ++s) { n_units += (rows(s) + 2 * spt - 1) / (2 * spt); longest = std::max(longest, n[s]); }
  const int units = n_units * Hkv;
  const int most_items = units <= c->n_sms ? c->n_sms / Hkv : 2 * units < 3 * c->n_sms ? SLOTS_PER_SM * c->n_sms / Hkv : n_units;     // as in attention_plan
  if (n_units > PLAN_UNITS || most_items <= n_units) return cut;       // nothing is cut and no merge launched whatever is said here
  // entities (units, tiles) by their number of pages
  struct Entity { float us; int times, pages; bool dbl; } ent[2][2 * PLAN_UNITS];
  short slot_of[2][4 * PLAN_UNITS];                    // open addressing; at most half full
  int n_ent[2] = {0, 0};
  float most_us[2] = {0.f, 0.f};
  memset(slot_of, 0xff, sizeof slot_of);
  auto add = [&](int list, int pages, bool dbl) {
    unsigned h = (unsigned)(pages * 2 + dbl) % (4 * PLAN_UNITS);
    while (slot_of[list][h] >= 0 && (ent[list][slot_of[list][h]].pages != pages || ent[list][slot_of[list][h]].dbl != dbl)) h = (h + 1) % (4 * PLAN_UNITS);
    if (slot_of[list][h] >= 0) { ++ent[list][slot_of[list][h]].times; return; }
    const float us = pages * (dbl ? PAIR_PAGE : SINGLE_PAGE);
    slot_of[list][h] = (short)n_ent[list];
    ent[list][n_ent[list]++] = Entity{us, 1, pages, dbl};
    most_us[list] = std::max(most_us[list], us);
  };
  struct Span { int nvis, loc; } span[3][PLAN_UNITS];  // of a block length's units, first tiles, second tiles: positions beyond n, local pages
  int spans = 0, spans_T = -1, tiles = 0;
  for (int s = 0; s < n_seqs; ++s) {
    const int k = ks ? ks[s] : k_all, T = rows(s);
    if (T != spans_T) {
      spans = 0; spans_T = T;
      auto seen = [&](int first, int last) {           // by slots first .. last
        int nvis = first < k ? std::min(last, k - 1) + 1 : 0, loc = 0;
        if (last >= k) { nvis = std::max(nvis, (last - k) / k + 1); loc = ((last - k) / k - (std::max(first, k) - k) / k + 1) * k; }
        return Span{nvis, (loc + PAGE - 1) / PAGE};
      };
      for (int r = 0; r < T; r += 2 * spt, ++spans) {
        span[0][spans] = seen(r, std::min(r + 2 * spt, T) - 1);
        span[1][spans] = seen(r, std::min(r + spt, T) - 1);
        span[2][spans] = r + spt < T ? seen(r + spt, std::min(r + 2 * spt, T) - 1) : Span{0, -1};
      }
    }
    for (int u = 0; u < spans; ++u) {
      const bool two = span[2][u].loc >= 0;
      auto pages = [&](const Span &x) { return (n[s] + x.nvis + PAGE - 1) / PAGE + x.loc; };
      add(0, pages(span[0][u]), two);
      add(1, pages(span[1][u]), false);
      if (two) add(1, pages(span[2][u]), false);
      tiles += two ? 2 : 1;
    }
  }
  float best = 1e30f;
  bool split = true;
  const bool may_cut = may_split(longest);
  for (int cnd = 0; cnd < 2 * CAND; cnd += 2) {        // (every other limit)
    const int list = cnd / CAND;
    const float lim = plan_limit(most_us[list], cnd % CAND);
    PlanCost cost{0, 0, 0, 0.f, 0.f};
    for (int e = 0; e < n_ent[list]; ++e) plan_add(cost, ent[list][e].us, lim, ent[list][e].dbl, ent[list][e].times);
    if (cost.items > most_items || cost.most > (may_cut ? MAX_SPLITS : 1)) continue;
    const float t = plan_time(cost, Hkv, c->n_sms);
    if (t < best) { best = t; split = cost.items > cost.live || (list == 1 && 2 * units > c->n_sms); }       // (single tiles beyond one wave need the larger grid)
  }
  // A cluster per tile, its pages shared evenly; on three quarters of the SMs at most, for on the others the projection behind the attention fills its
  // rings (8B-class step of 272 rows, clusters of two on 144 SMs: attention 15.9 -> 12.7 us, the O projection 14.9 -> 18).
  const int places = mixed ? 2 * ((n_units + 3) / 4 * 4) : tiles;      // items of the launch (see attention_plan)
  if (split) best += 1.5f;                               // (the boundary in front of the merge kernel)
  StepAttention pick = split ? cut : uncut;
  for (int size = 2; size <= MAX_CLUSTER && size * 16 <= c->cfg.head_dim; size *= 2) {
    const float t = std::ceil(most_us[1] / SINGLE_PAGE / size) * SINGLE_PAGE + OVERHEAD + CLUSTER_MERGE;
    if (places * Hkv <= c->max_clusters[size] && 4 * places * Hkv * size <= 3 * c->n_sms && t < best - 0.3f) { best = t; pick = {false, size}; }
  }
  return pick;
}

attn_tc::Args attention_args(const tidar_ctx *c, const AttnMaps &m, const KvGeom &g, bf16 *O) {
  const tidar_config &cf = c->cfg;
  attn_tc::Args a{};
  a.G = cf.n_q_heads / cf.n_kv_heads; a.Hq = cf.n_q_heads; a.Hkv = cf.n_kv_heads; a.spt = 128 / a.G;
  a.nvis = c->meta.nvis; a.loc0 = c->meta.loc0; a.nloc = c->meta.nloc;
  a.page_table = g.page_table; a.pages_per_seq = g.pages_per_seq;
  a.page_base_k = m.page_base_k; a.page_base_v = m.page_base_v;
  a.scale_log2 = 1.4426950408889634f / sqrtf((float)cf.head_dim);
  a.O = O; a.part_O = c->attn_part_O; a.part_ml = c->attn_part_ml; a.status = c->d_status;
  a.tile_count = c->count_tiles ? c->d_tl + 2 * tidar_ctx::TL_MAX : nullptr;
  return a;
}
// One CTA per item, or (cluster > 1) a cluster of CTAs per item.
template <int STREAMS, bool DIRECT, bool AHEAD = false>
void launch_attention_kernel(tidar_ctx *c, int grid, const AttnMaps &m, const attn_tc::Args &a, int cluster = 1) {
  Launch l(c, TIDAR_TC_ATTN);
  const int threads = attn_tc::threads(STREAMS);
  if constexpr (STREAMS == 2) {
    if (cluster > 1) {
      if (c->cfg.head_dim == 128)
        launch_pdl_cluster(cluster, attn_tc::attn_tc_kernel<128, 2, DIRECT, AHEAD, true>, grid * cluster, threads, attn_tc::Smem<128, 2, true>::TOTAL, c->stream, *m.q, *m.k,
                           *m.v, *m.kloc, *m.vloc, a, l.tl);
      else
        launch_pdl_cluster(cluster, attn_tc::attn_tc_kernel<64, 2, DIRECT, AHEAD, true>, grid * cluster, threads, attn_tc::Smem<64, 2, true>::TOTAL, c->stream, *m.q, *m.k,
                           *m.v, *m.kloc, *m.vloc, a, l.tl);
      return;
    }
  }
  if (c->cfg.head_dim == 128)
    launch_pdl(attn_tc::attn_tc_kernel<128, STREAMS, DIRECT, AHEAD, false>, grid, threads, attn_tc::Smem<128, STREAMS>::TOTAL, c->stream, *m.q, *m.k, *m.v, *m.kloc, *m.vloc, a, l.tl);
  else
    launch_pdl(attn_tc::attn_tc_kernel<64, STREAMS, DIRECT, AHEAD, false>, grid, threads, attn_tc::Smem<64, STREAMS>::TOTAL, c->stream, *m.q, *m.k, *m.v, *m.kloc, *m.vloc, a, l.tl);
}

template <bool DIRECT>
void launch_attention_merge(tidar_ctx *c, int tiles, const attn_tc::Args &a) {
  Launch l(c, TIDAR_TC_ATTN);
  const int blocks = tiles * (c->cfg.head_dim / 16);
  if (c->cfg.head_dim == 128) launch_pdl(attn_tc::attn_combine_kernel<128, DIRECT>, blocks, 256, 0, c->stream, a, l.tl);
  else launch_pdl(attn_tc::attn_combine_kernel<64, DIRECT>, blocks, 256, 0, c->stream, a, l.tl);
}

bool merges(const attn_tc::PlanArgs &p) { return p.max_items > p.n_units && p.max_pieces > 1; }
void note_route(tidar_ctx *c, const attn_tc::PlanArgs &p) { c->route = {p.singles ? c->attn_cluster : 1, merges(p), p.n_units <= attn_tc::PLAN_UNITS ? p.n_units : 0}; }

// Attention of the pass that plan p was made for (the plan itself is in device memory by then).  early: see attn_tc::Args; ahead: see attn_tc_kernel.
void launch_attention_tc(tidar_ctx *c, const attn_tc::PlanArgs &p, const AttnMaps &m, const KvGeom &g, bf16 *O, bool early, bool ahead) {
  attn_tc::Args a = attention_args(c, m, g, O);
  a.items = p.items; a.tiles = p.tiles;
  a.early = early ? 1 : 0;
  const int cluster = p.singles ? c->attn_cluster : 1;
  if (early && ahead) launch_attention_kernel<2, false, true>(c, p.max_items * p.Hkv, m, a, cluster); else launch_attention_kernel<2, false>(c, p.max_items * p.Hkv, m, a, cluster);
  if (merges(p)) launch_attention_merge<false>(c, 2 * p.n_units * p.Hkv, a);
}

// How a stand-alone call goes without a plan, every CTA working out its own item: streams per CTA (0 = planned) and items per query tile.
// n_pages: pages a sequence may have (its length is on the device).  The plan kernel costs 4.5 us, which a pass pays once for all
// layers but such a call alone; cutting a key range into p items saves (1 - 1/p) of 0.56 us per page and costs about 6 + 0.3 p us
// (partial results, merge kernel).
//   Where every tile may have as many SMs as it can use, sqrt(0.56 n_pages / 0.3), there is nothing to distribute: uncut up to 15 pages, cut
//     evenly beyond (one sequence, k = 8, 32/8 heads of 128: 14.4 us uncut and 15.8 cut at 15 pages, 15.5 and 15.8 at 17, 16.4 and 16.1 at
//     19; planned 18 - 18.7).
//   Otherwise uncut while that is faster than planned: measured equal at 24 pages for four SMs per tile, 31 for two; the line
//     lies a little below.  (k = 16, 1 k positions, 72 tiles: 18.9 us planned, 13.6 uncut.)
//   With one to two tiles per SM, one stream per CTA and two CTAs per SM: one wave, where the plan's CTAs, which hold an SM each, need
//     two.  Four sequences of 1 k positions there (288 tiles): 42.1 us planned, 25.7 this way, at 9 k 175 and 148; but a plan evens
//     out ragged lengths, which pays from about 60 pages on (lengths between 2 k and 4 k: 53.9 planned, 58.1 not).
struct DirectPlan { int streams, pieces, cluster; };
DirectPlan attention_direct(const tidar_ctx *c, int n_seqs, int k, int n_pages) {
  const int spt = 128 / (c->cfg.n_q_heads / c->cfg.n_kv_heads);
  const long long tiles = (long long)n_seqs * ((k * (k + 1) + spt - 1) / spt) * c->cfg.n_kv_heads;
  if (tiles > c->n_sms) return {tiles <= 2 * c->n_sms && n_pages <= 40 ? 1 : 0, 1, 1};
  const int most = std::min<int>(attn_tc::MAX_SPLITS, c->n_sms / (int)tiles);
  const int pieces = (int)sqrt(1.9 * n_pages);
  if (n_pages <= (pieces <= most ? 15 : 19 + 12 / most)) {
    DirectPlan pick{2, 1, 1};
    float best = n_pages * attn_tc::SINGLE_PAGE - 0.3f;
    for (int size = 2; size <= attn_tc::MAX_CLUSTER && size * 16 <= c->cfg.head_dim; size *= 2) {
      const float t = (n_pages + size - 1) / size * attn_tc::SINGLE_PAGE + attn_tc::CLUSTER_MERGE;
      if (tiles <= c->max_clusters[size] && t < best) { best = t; pick.cluster = size; }
    }
    return pick;
  }
  return {pieces <= most ? 2 : 0, pieces, 1};
}

void launch_attention(tidar_ctx *c, const bf16 *Q, const bf16 *Kp, const bf16 *Vp, const KvGeom &g, const bf16 *Kl,
                      const bf16 *Vl, bf16 *O, int R) {
  Launch l(c, TIDAR_TC_ATTN);
  const float scale = 1.0f / sqrtf((float)c->cfg.head_dim);
  dim3 grid(R, c->cfg.n_q_heads);
  if (c->cfg.head_dim == 128)
    attn_replay_kernel<128><<<grid, 32, 0, c->stream>>>(Q, Kp, Vp, g, c->meta, Kl, Vl, O, c->cfg.n_q_heads, scale);
  else
    attn_replay_kernel<64><<<grid, 32, 0, c->stream>>>(Q, Kp, Vp, g, c->meta, Kl, Vl, O, c->cfg.n_q_heads, scale);
}

// How the norm of R rows of d floats with S fp32 partial results each is launched.
// Behind a projection of many rows the blocks would all crowd onto the SMs that run out of work first (5.6 instead of
// 3.6 us at 272 rows); claiming a share of the shared memory spreads them evenly.  With few rows they must leave room
// for the next projection's CTAs.
// Bulk copies where a row and its partial results are many bytes and every SM has one or two rows (measured: 82 KB 1.4 times as fast; 30 KB, 272 rows of
// 1536 with four slabs, 1.8 -> 2.3 us; 16 KB, 1152 rows of 4096 without slabs, 5.5 -> 6.4; 20 rows of 82 KB no difference).
struct NormPlan { bool bulk; size_t smem; };
NormPlan norm_plan(int n_sms, int R, int d, int S, bool fp32_slabs) {
  const int per_sm = (R + n_sms - 1) / n_sms;
  if (R <= gemm_tc::SMALL_ROWS || per_sm > 4) return {false, 0};
  const size_t share = (size_t)(NORM_SMEM / per_sm) & ~(size_t)1023, bytes = (size_t)(S + 1) * d * sizeof(float);
  return {fp32_slabs && R <= gemm_tc::MAX_ROWS && per_sm <= 2 && bytes >= 48 * 1024 && bytes <= share, share};
}

// partials: split-K slabs of the previous projection, bf16 on the tensor-core path, fp32 on the replay path
template <typename SLAB>
void launch_norm_as(tidar_ctx *c, int R, const SLAB *partials, int S, size_t stride, const bf16 *gain) {
  Launch l(c, TIDAR_TC_NORM);
  const int d = c->cfg.d_model, nv = (d + 2047) / 2048;
  const NormPlan plan = c->cfg.impl == 0 ? norm_plan(c->n_sms, R, d, S, std::is_same_v<SLAB, float>) : NormPlan{false, 0};
  if constexpr (std::is_same_v<SLAB, float>) {
    if (plan.bulk) {
      auto bulk = [&](auto kernel) { launch_pdl(kernel, R, 512, plan.smem, c->stream, c->X, partials, S, stride, gain, c->cfg.rms_eps, d, c->A, c->d_status, l.tl); };
      if (nv <= 1) bulk(rmsnorm_bulk_kernel<512, 1>);
      else if (nv <= 2) bulk(rmsnorm_bulk_kernel<512, 2>);
      else if (nv <= 3) bulk(rmsnorm_bulk_kernel<512, 3>);
      else bulk(rmsnorm_bulk_kernel<512, 6>);
      return;
    }
  }
  auto go = [&](auto kernel) { launch_pdl(kernel, R, 512, plan.smem, c->stream, c->X, partials, S, stride, gain, c->cfg.rms_eps, d, c->A, l.tl); };
  auto by_width = [&](auto slabs, auto walk) {
    constexpr int SL = decltype(slabs)::value;
    constexpr bool WK = decltype(walk)::value;
    if (nv <= 1) go(rmsnorm_reduce_kernel<512, 1, SL, WK, SLAB>);
    else if (nv <= 2) go(rmsnorm_reduce_kernel<512, 2, SL, WK, SLAB>);
    else if (nv <= 3) go(rmsnorm_reduce_kernel<512, 3, SL, WK, SLAB>);
    else go(rmsnorm_reduce_kernel<512, 6, SL, WK, SLAB>);
  };
  auto by_rows = [&](auto slabs) { if (R <= gemm_tc::SMALL_ROWS) by_width(slabs, std::true_type()); else by_width(slabs, std::false_type()); };
  if (S <= 1) by_rows(std::integral_constant<int, 1>()); else by_rows(std::integral_constant<int, MAX_SLABS>());
}
void launch_norm(tidar_ctx *c, int R, const float *partials, int S, size_t stride, const bf16 *gain) {
  if (c->cfg.impl == 0 && c->slab_bf16) launch_norm_as<bf16>(c, R, (const bf16 *)partials, S, stride, gain);
  else launch_norm_as<float>(c, R, partials, S, stride, gain);
}

// The transformer stack over R assembled rows (metadata and X already filled).
// with_head: run final norm + LM head + per-row argmax.
// Extra LM-head input rows that mix two final-normed rows each (beta < 1; see mix_rows_kernel).
struct MixRows { int n = 0, k = 1, a0 = 0, a_seq = 0, a_j = 0, b0 = 0, b_seq = 0, b_j = 0; StepLayout lay{nullptr, nullptr, nullptr, 0}; };

// head_row0: the LM head (with_head) runs on rows [head_row0, R) only, followed by the mixed rows; the
// argmax ids and the logits dump are indexed from head_row0.
// step: a decode step (its rows see at most k_max positions more than are cached).
int forward_rows(tidar_ctx *c, int R, bool with_head, int rows_per_group, const MixRows &mix = MixRows(), int head_row0 = 0, bool step = false) {
  const tidar_config &cf = c->cfg;
  const int d = cf.d_model, hd = cf.head_dim, Hq = cf.n_q_heads, Hkv = cf.n_kv_heads;
  const KvGeom g = geom(c);
  const attn_tc::PlanArgs plan = cf.impl == 0 ? attention_plan(c, R, rows_per_group) : attn_tc::PlanArgs{};
  {
    Launch l(c, TIDAR_TC_ROPE);
    const int n = R * (hd / 2);
    launch_pdl(pass_setup_kernel, (n + 255) / 256 + (plan.tiles ? 1 : 0), 256, 0, c->stream, c->meta, R, hd / 2, (double)cf.rope_theta, c->rope_cos,
                 c->rope_sin, plan, l.tl);
  }
  int S = 0; size_t stride = 0;          // pending partials of the previous down projection
  const bool tc = cf.impl == 0, few = R <= gemm_tc::SMALL_ROWS;
  const int RA = c->R_cap;               // allocated rows of the activation buffers
  int rc;
  for (int l = 0; l < cf.n_layers; ++l) {
    bf16 *Kp = c->kv + (size_t)(2 * l) * c->pool_stride, *Vp = Kp + c->pool_stride;
    launch_norm(c, R, c->partials, S, stride, c->attn_norm[l]);
    if (c->dbg_hidden)
      CUDA_TRY(c, cudaMemcpyAsync(c->dbg_hidden + (size_t)l * c->R_cap * d, c->X, (size_t)R * d * sizeof(float),
                                  cudaMemcpyDeviceToDevice, c->stream));
    if ((rc = gemm_partials(c, c->A, RA, c->wqkv[l], tc ? &c->tm_wqkv[l] : nullptr, R, c->n_qkv, d, c->partials, &S, &stride, TIDAR_TC_GEMM))) return rc;
    {
      Launch ll(c, TIDAR_TC_ROPE);
      const int rope_chunks = ((Hq + 2 * Hkv) * (hd / 8) + 255) / 256;
      const bf16 *bias_l = c->bqkv.empty() ? nullptr : c->bqkv[l], *qn_l = c->q_norm.empty() ? nullptr : c->q_norm[l],
                 *kn_l = c->k_norm.empty() ? nullptr : c->k_norm[l];
      auto rope = [&](auto kernel, auto *partials) {
        launch_pdl(kernel, dim3(R, rope_chunks), 256, 0, c->stream, partials, S, stride, Hq, Hkv, hd, c->meta, c->rope_cos, c->rope_sin, g, c->Q, Kp, Vp,
                   c->Kloc, c->Vloc, bias_l, qn_l, kn_l, cf.rms_eps, l > 0 && few ? 1 : 0, ll.tl);
      };
      const bool walk = tc && l > 0 && few;                  // (the first layer's attention lies between the metadata's writer and this kernel)
      if (tc && c->slab_bf16) rope(rope_kv_kernel<MAX_SLABS, false, bf16>, (const bf16 *)c->partials);
      else if (S <= 1) walk ? rope(rope_kv_kernel<1, true, float>, (const float *)c->partials) : rope(rope_kv_kernel<1, false, float>, (const float *)c->partials);
      else walk ? rope(rope_kv_kernel<MAX_SLABS, true, float>, (const float *)c->partials) : rope(rope_kv_kernel<MAX_SLABS, false, float>, (const float *)c->partials);
    }
    if (tc) {
      AttnMaps am{&c->tm_q, &c->tm_kv, &c->tm_kv, &c->tm_kloc, &c->tm_vloc, (2 * l) * c->n_pages, (2 * l + 1) * c->n_pages};
      launch_attention_tc(c, plan, am, g, c->O, true, step && few);     // behind the RoPE kernel
    } else {
      launch_attention(c, c->Q, Kp, Vp, g, c->Kloc, c->Vloc, c->O, R);
    }
    if ((rc = gemm_partials(c, c->O, RA, c->wo[l], tc ? &c->tm_wo[l] : nullptr, R, d, Hq * hd, c->partials, &S, &stride, TIDAR_TC_GEMM, c->X))) return rc;
    launch_norm(c, R, c->partials, S, stride, c->ffn_norm[l]);
    if (tc) {
      if ((rc = gemm_tc_launch(c, gemm_tc::MODE_SWIGLU, c->A, RA, c->tm_wgu[l], R, 2 * cf.d_ffn, d, TIDAR_TC_GEMM, nullptr, nullptr))) return rc;
    } else {
      if ((rc = gemm_partials(c, c->A, RA, c->wgu[l], nullptr, R, 2 * cf.d_ffn, d, c->partials, &S, &stride, TIDAR_TC_GEMM))) return rc;
      Launch ll(c, TIDAR_TC_GEMM);
      const size_t n = (size_t)R * cf.d_ffn;
      swiglu_kernel<<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(c->partials, R, cf.d_ffn, c->H);
    }
    if ((rc = gemm_partials(c, c->H, RA, c->wdown[l], tc ? &c->tm_wdown[l] : nullptr, R, d, cf.d_ffn, c->partials, &S, &stride, TIDAR_TC_GEMM, c->X))) return rc;
  }
  launch_norm(c, R, c->partials, S, stride, c->final_norm);
  if (c->dbg_hidden)
    CUDA_TRY(c, cudaMemcpyAsync(c->dbg_hidden + (size_t)cf.n_layers * c->R_cap * d, c->X, (size_t)R * d * sizeof(float),
                                cudaMemcpyDeviceToDevice, c->stream));
  if (with_head && mix.n > 0) {            // rows R .. R + mix.n - 1 of the LM head's input
    Launch lm(c, TIDAR_TC_NORM);
    launch_pdl(mix_rows_kernel, mix.n, 256, 0, c->stream, c->A, d, cf.beta, mix.k, mix.a0, mix.a_seq, mix.a_j, mix.b0, mix.b_seq, mix.b_j, mix.lay, R,
                 cf.temperature > 0.f ? c->meta.skey : (uint32_t *)nullptr, lm.tl);
    R += mix.n;
  }
  const bf16 *Ah = c->A + (size_t)head_row0 * d;           // first row of the LM head's input
  c->head_row0 = head_row0;
  const float inv_temp = cf.temperature > 0.f ? 1.0f / cf.temperature : 0.f;
  const int Rh = R - head_row0;
  if (with_head && Rh > c->R_head) return fail(c, TIDAR_ECAPACITY, "%d rows for the LM head exceed the context's %d", Rh, c->R_head);
  if (with_head && tc) {
    // with one row block every CTA leaves a candidate for every row; with several it may meet only some of them
    const bool one_block = Rh <= gemm_tc::MAX_ROWS;
    const int G = lm_head_ctas(c, Rh, cf.vocab) * 4;
    if (!one_block) CUDA_TRY(c, cudaMemsetAsync(c->cand_idx, 0xff, (size_t)G * Rh * sizeof(int32_t), c->stream));
    if ((rc = gemm_tc_launch(c, gemm_tc::MODE_ARGMAX, Ah, RA - head_row0, c->tm_lm, Rh, cf.vocab, d, TIDAR_TC_LMHEAD, nullptr, nullptr))) return rc;
    Launch ll(c, TIDAR_TC_LMHEAD);
    launch_pdl(argmax_merge_kernel, (Rh * 32 + 255) / 256, 256, 0, c->stream, c->cand_val, c->cand_idx, G, Rh, c->d_arg_val, c->d_arg_idx, ll.tl);
  } else if (with_head) {
    for (int v0 = 0; v0 < cf.vocab; v0 += c->lm_chunk) {
      const int nc = std::min(c->lm_chunk, cf.vocab - v0);
      if ((rc = gemm_partials(c, Ah, RA - head_row0, c->lm_head + (size_t)v0 * d, nullptr, Rh, nc, d, c->partials, &S, &stride, TIDAR_TC_LMHEAD))) return rc;
      Launch ll(c, TIDAR_TC_LMHEAD);
      argmax_chunk_kernel<<<Rh, 256, 0, c->stream>>>(c->partials, nc, nc, v0, v0 == 0, c->d_arg_val, c->d_arg_idx, c->dbg_logits, cf.vocab, inv_temp,
                                                     c->meta.skey + head_row0);
    }
  }
  CUDA_TRY(c, cudaGetLastError());
  return TIDAR_OK;
}

// Driver entry point for tensor-map encoding (resolved through the runtime so that the
// library has no link-time dependency on the driver), tensor maps of every weight
// matrix, kernel attributes.
int init_tensor_core_path(tidar_ctx *c) {
  const tidar_config &cf = c->cfg;
  int dev = 0;
  CUDA_TRY(c, cudaGetDevice(&dev));
  int major = 0, minor = 0;                       // (cudaGetDeviceProperties takes milliseconds)
  CUDA_TRY(c, cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
  CUDA_TRY(c, cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev));
  CUDA_TRY(c, cudaDeviceGetAttribute(&c->n_sms, cudaDevAttrMultiProcessorCount, dev));
  if (major != 10) return fail(c, TIDAR_ECUDA, "the tensor-core path needs an sm_100 device, found sm_%d%d", major, minor);
  if (c->n_sms > MAX_SMS) return fail(c, TIDAR_ECUDA, "%d SMs; scratch is sized for %d", c->n_sms, MAX_SMS);
  void *fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  CUDA_TRY(c, cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres));
  if (!fn || qres != cudaDriverEntryPointSuccess) return fail(c, TIDAR_ECUDA, "cuTensorMapEncodeTiled is not available in this driver");
  c->encode = (gemm_tc::EncodeTiledFn)fn;
  const int d = cf.d_model, qo = cf.n_q_heads * cf.head_dim;
  auto enc = [&](tidar_ctx::WMap *tm, const void *p, int rows, int cols) { return encode_weights(c, tm, p, rows, cols); };
  c->tm_wqkv.resize(cf.n_layers); c->tm_wo.resize(cf.n_layers); c->tm_wgu.resize(cf.n_layers); c->tm_wdown.resize(cf.n_layers);
  bool ok = enc(&c->tm_lm, c->lm_head, cf.vocab, d);
  for (int l = 0; l < cf.n_layers && ok; ++l)
    ok = enc(&c->tm_wqkv[l], c->wqkv[l], c->n_qkv, d) && enc(&c->tm_wo[l], c->wo[l], d, qo) &&
         enc(&c->tm_wgu[l], c->wgu[l], 2 * cf.d_ffn, d) && enc(&c->tm_wdown[l], c->wdown[l], d, cf.d_ffn);
  if (!ok) return fail(c, TIDAR_ECUDA, "cuTensorMapEncodeTiled failed for a weight matrix (pointers must be 16-byte aligned)");
  {
    const size_t nloc = (size_t)std::max(cf.max_batch * cf.k_max * cf.k_max, cf.k_max);
    if (!encode_q_map(c, &c->tm_q, c->Q, c->R_cap) || !encode_pages_map(c, &c->tm_kv, c->kv, (long long)cf.n_layers * 2 * c->n_pages) ||
        !encode_local_map(c, &c->tm_kloc, c->Kloc, (long long)nloc) || !encode_local_map(c, &c->tm_vloc, c->Vloc, (long long)nloc))
      return fail(c, TIDAR_ECUDA, "cuTensorMapEncodeTiled failed for an attention operand");
    // The PV product multiplies masked keys' V rows by an exact zero, so whatever the
    // kernel may load (unwritten cache slots of a page, unwritten local rows) must be finite.
    CUDA_TRY(c, cudaMemsetAsync(c->kv, 0, (size_t)cf.n_layers * 2 * c->pool_stride * sizeof(bf16), c->stream));
    CUDA_TRY(c, cudaMemsetAsync(c->Kloc, 0, nloc * cf.n_kv_heads * cf.head_dim * sizeof(bf16), c->stream));
    CUDA_TRY(c, cudaMemsetAsync(c->Vloc, 0, nloc * cf.n_kv_heads * cf.head_dim * sizeof(bf16), c->stream));
    auto smem = [](const void *f, int bytes) { return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); };
    CUDA_TRY(c, smem((const void *)attn_tc::attn_tc_kernel<128, 2, false, false, false>, attn_tc::Smem<128, 2>::TOTAL));
    CUDA_TRY(c, smem((const void *)attn_tc::attn_tc_kernel<128, 2, false, true, false>, attn_tc::Smem<128, 2>::TOTAL));
    CUDA_TRY(c, smem((const void *)attn_tc::attn_tc_kernel<64, 2, false, false, false>, attn_tc::Smem<64, 2>::TOTAL));
    CUDA_TRY(c, smem((const void *)attn_tc::attn_tc_kernel<64, 2, false, true, false>, attn_tc::Smem<64, 2>::TOTAL));
    CUDA_TRY(c, smem((const void *)attn_tc::attn_tc_kernel<128, 2, true, false, false>, attn_tc::Smem<128, 2>::TOTAL));
    CUDA_TRY(c, smem((const void *)attn_tc::attn_tc_kernel<64, 2, true, false, false>, attn_tc::Smem<64, 2>::TOTAL));
    auto clusters = [&](auto kernel_128, auto kernel_64) {
      const void *f = cf.head_dim == 128 ? (const void *)kernel_128 : (const void *)kernel_64;
      const int bytes = cf.head_dim == 128 ? attn_tc::Smem<128, 2, true>::TOTAL : attn_tc::Smem<64, 2, true>::TOTAL;
      return smem(f, bytes);
    };
    CUDA_TRY(c, clusters(attn_tc::attn_tc_kernel<128, 2, false, false, true>, attn_tc::attn_tc_kernel<64, 2, false, false, true>));
    CUDA_TRY(c, clusters(attn_tc::attn_tc_kernel<128, 2, false, true, true>, attn_tc::attn_tc_kernel<64, 2, false, true, true>));
    CUDA_TRY(c, clusters(attn_tc::attn_tc_kernel<128, 2, true, false, true>, attn_tc::attn_tc_kernel<64, 2, true, false, true>));
    for (int size = 2; size <= attn_tc::MAX_CLUSTER && size * 16 <= cf.head_dim; size *= 2) {
      cudaLaunchConfig_t lc{};
      lc.gridDim = dim3(size); lc.blockDim = dim3(attn_tc::threads(2));
      lc.dynamicSmemBytes = cf.head_dim == 128 ? attn_tc::Smem<128, 2, true>::TOTAL : attn_tc::Smem<64, 2, true>::TOTAL;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = size; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
      lc.attrs = at; lc.numAttrs = 1;
      CUDA_TRY(c, cudaOccupancyMaxActiveClusters(&c->max_clusters[size], cf.head_dim == 128 ? (const void *)attn_tc::attn_tc_kernel<128, 2, false, false, true>
                                                                                            : (const void *)attn_tc::attn_tc_kernel<64, 2, false, false, true>, &lc));
    }
    CUDA_TRY(c, smem((const void *)attn_tc::attn_tc_kernel<128, 1, true, false, false>, attn_tc::Smem<128, 1>::TOTAL));
    CUDA_TRY(c, smem((const void *)attn_tc::attn_tc_kernel<64, 1, true, false, false>, attn_tc::Smem<64, 1>::TOTAL));
  }
  {
    auto max_smem_split = [&](const void *f) { return cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared); };
    const void *kernels[] = {(const void *)assemble_step_kernel, (const void *)pass_setup_kernel, (const void *)attn_meta_plan_kernel,
                             (const void *)rope_kv_kernel<1, false, float>, (const void *)rope_kv_kernel<MAX_SLABS, false, float>, (const void *)rope_kv_kernel<MAX_SLABS, false, bf16>,
                             (const void *)rope_kv_kernel<1, true, float>, (const void *)rope_kv_kernel<MAX_SLABS, true, float>,
                             (const void *)swiglu_slab_kernel<float>, (const void *)swiglu_slab_kernel<bf16>,
                             (const void *)attn_tc::attn_combine_kernel<128, false>, (const void *)attn_tc::attn_combine_kernel<64, false>,
                             (const void *)attn_tc::attn_combine_kernel<128, true>, (const void *)attn_tc::attn_combine_kernel<64, true>,
                             (const void *)mix_rows_kernel, (const void *)argmax_merge_kernel, (const void *)verify_select_kernel, (const void *)stage_step_kernel};
    for (const void *f : kernels) CUDA_TRY(c, max_smem_split(f));
    std::vector<const void *> norms = {(const void *)rmsnorm_bulk_kernel<512, 1>, (const void *)rmsnorm_bulk_kernel<512, 2>, (const void *)rmsnorm_bulk_kernel<512, 3>,
                                       (const void *)rmsnorm_bulk_kernel<512, 6>};
    auto add_norms = [&](auto slabs, auto slab) {
      constexpr int SL = decltype(slabs)::value;
      using T = decltype(slab);
      for (const void *f : {(const void *)rmsnorm_reduce_kernel<512, 1, SL, false, T>, (const void *)rmsnorm_reduce_kernel<512, 1, SL, true, T>,
                            (const void *)rmsnorm_reduce_kernel<512, 2, SL, false, T>, (const void *)rmsnorm_reduce_kernel<512, 2, SL, true, T>,
                            (const void *)rmsnorm_reduce_kernel<512, 3, SL, false, T>, (const void *)rmsnorm_reduce_kernel<512, 3, SL, true, T>,
                            (const void *)rmsnorm_reduce_kernel<512, 6, SL, false, T>, (const void *)rmsnorm_reduce_kernel<512, 6, SL, true, T>}) norms.push_back(f);
    };
    add_norms(std::integral_constant<int, 1>(), float()); add_norms(std::integral_constant<int, 1>(), bf16());
    add_norms(std::integral_constant<int, MAX_SLABS>(), float()); add_norms(std::integral_constant<int, MAX_SLABS>(), bf16());
    for (const void *f : norms) {
      CUDA_TRY(c, max_smem_split(f));
      CUDA_TRY(c, cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, NORM_SMEM));
    }
    CUDA_TRY(c, max_smem_split((const void *)attn_tc::attn_tc_kernel<128, 1, true, false, false>));
    CUDA_TRY(c, max_smem_split((const void *)attn_tc::attn_tc_kernel<64, 1, true, false, false>));
  }
  const int max_smem = gemm_tc::SMEM_BUDGET + 1024;
  CUDA_TRY(c, cudaFuncSetAttribute(gemm_tc::gemm_tc_kernel<gemm_tc::MODE_SLAB, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem));
  CUDA_TRY(c, cudaFuncSetAttribute(gemm_tc::gemm_tc_kernel<gemm_tc::MODE_SWIGLU, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem));
  CUDA_TRY(c, cudaFuncSetAttribute(gemm_tc::gemm_tc_kernel<gemm_tc::MODE_SLAB, true>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
  CUDA_TRY(c, cudaFuncSetAttribute(gemm_tc::gemm_tc_kernel<gemm_tc::MODE_SWIGLU, true>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
  CUDA_TRY(c, cudaFuncSetAttribute(gemm_tc::gemm_tc_kernel<gemm_tc::MODE_SLAB>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem));
  CUDA_TRY(c, cudaFuncSetAttribute(gemm_tc::gemm_tc_kernel<gemm_tc::MODE_SWIGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem));
  CUDA_TRY(c, cudaFuncSetAttribute(gemm_tc::gemm_tc_kernel<gemm_tc::MODE_ARGMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem));
  CUDA_TRY(c, cudaFuncSetAttribute(gemm_tc::gemm_tc_kernel<gemm_tc::MODE_LSE>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem));
  CUDA_TRY(c, cudaFuncSetAttribute(gemm_tc::gemm_tc_kernel<gemm_tc::MODE_SAMPLE>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem));
  return TIDAR_OK;
}

int device_timeout(tidar_ctx *c, int st) {
  return fail(c, TIDAR_EDEVICE_TIMEOUT, "a bounded device-side wait gave up (status %d); results of this call are invalid", st);
}

// Reads the device status word and turns a device-side timeout into an error code.
int check_device_status(tidar_ctx *c) {
  if (c->cfg.impl != 0) return TIDAR_OK;
  int st = 0;
  CUDA_TRY(c, cudaMemcpyAsync(&st, c->d_status, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  if (st) {
    cudaMemsetAsync(c->d_status, 0, sizeof(int), c->stream);
    return device_timeout(c, st);
  }
  return TIDAR_OK;
}

// Returns a sequence slot's pages to the pool and marks it as not prefilled.
void release_sequence(tidar_ctx *c, int seq) {
  SeqState &s = c->seqs[seq];
  for (int p : s.pages) c->free_pages.push_back(p);
  s.pages.clear(); s.active = false; s.n = 0;
}

int ensure_pages(tidar_ctx *c, int seq, int upto_positions) {
  SeqState &s = c->seqs[seq];
  const int need = (upto_positions + c->cfg.page_size - 1) / c->cfg.page_size;
  if (need > c->pages_per_seq) return fail(c, TIDAR_ECAPACITY, "sequence %d needs %d pages, limit %d", seq, need, c->pages_per_seq);
  if ((int)s.pages.size() >= need) return TIDAR_OK;
  // The copy reads a pinned mirror that nothing else writes at these entries until the sequence is
  // released and prefilled again (which only happens with no step in flight), so it needs no wait.
  int32_t *row = c->h_page_table + (size_t)seq * c->pages_per_seq;
  const int have = (int)s.pages.size();
  while ((int)s.pages.size() < need) {
    if (c->free_pages.empty()) return fail(c, TIDAR_ECAPACITY, "KV page pool exhausted");
    row[s.pages.size()] = c->free_pages.back();
    s.pages.push_back(c->free_pages.back());
    c->free_pages.pop_back();
  }
  CUDA_TRY(c, cudaMemcpyAsync(c->d_page_table + (size_t)seq * c->pages_per_seq + have, row + have, (size_t)(need - have) * sizeof(int),
                              cudaMemcpyHostToDevice, c->stream));
  return TIDAR_OK;
}

StepIo step_io(const tidar_ctx *c) {
  StepIo io;
  io.turn = c->d_status + 16; io.blocks_done = c->d_status + 32; io.status = c->d_status;
  for (int sl = 0; sl < 2; ++sl) { io.in[sl] = c->h_stage2[sl]; io.out[sl] = c->h_out2[sl]; io.done[sl] = c->h_done2[sl]; }
  io.max_batch = c->cfg.max_batch;
  return io;
}

// Enqueues the kernels of one decode step (its inputs are in the slot's pinned staging).
// key.k: block length of this step; key.ar: plain autoregressive step (the causal section alone).
// key.mixed_R > 0: the listed sequences use different block lengths (layout staged in h_lay, mixed_R rows in all).
// key.mixed_K: the sum of those block lengths (= verified positions, one mixed row each when beta < 1).
int record_step(tidar_ctx *c, const tidar_ctx::StepKey &key) {
  const tidar_config &cf = c->cfg;
  const int n_seqs = key.n_seqs, k = key.k, n_blocks = key.ar ? 0 : k;
  const int T = k * (n_blocks + 1), R = key.mixed_R > 0 ? key.mixed_R : n_seqs * T;
  StepLayout lay{nullptr, nullptr, nullptr, n_seqs};
  if (key.mixed_R > 0) { lay.k = c->d_step_k; lay.off = c->d_step_off; lay.loc = c->d_step_loc; }
  c->split_keys = key.split; c->attn_cluster = key.cluster;
  c->mixed_units = key.units;
  if (c->timeline) {
    c->tl_n = 0; c->tl_cls.clear();
    CUDA_TRY(c, cudaMemsetAsync(c->d_tl, 0, 2 * tidar_ctx::TL_MAX * sizeof(unsigned long long), c->stream));
  }
  const StepIo io = step_io(c);
  {
    Launch l(c, TIDAR_TC_EMBED);
    launch_pdl(stage_step_kernel, 1, 256, 0, c->stream, io, n_seqs, c->d_step_seqs, c->d_forced, c->h_lay, c->d_step_k,
               key.mixed_R > 0 ? 3 * (cf.max_batch + 1) : 0, c->R_head + cf.max_batch, key.units, l.tl);
  }
  {
    Launch l(c, TIDAR_TC_EMBED);
    launch_pdl(assemble_step_kernel, R, 256, 0, c->stream, c->meta, c->d_step_seqs, c->d_seq_len, c->d_block, c->d_blk_len, k, n_blocks, lay, cf.k_max,
               cf.mask_token_id, c->d_step_n, c->embed, cf.d_model, c->X, cf.temperature > 0.f ? 1 : 0, (unsigned long long)cf.sample_seed, l.tl);
  }
  // beta < 1: the verified prediction of causal slot j mixes its row with the first slot of block j
  MixRows mix;
  if (cf.beta < 1.0f && !key.ar) {
    if (key.mixed_R > 0) { mix.n = key.mixed_K; mix.lay = lay; }
    else { mix.n = n_seqs * k; mix.k = k; mix.a0 = 0; mix.a_seq = T; mix.a_j = 1; mix.b0 = k; mix.b_seq = T; mix.b_j = k; }
  }
  if (int rc = forward_rows(c, R, true, key.mixed_R > 0 ? 0 : T, mix, 0, true)) return rc;
  {
    Launch l(c, TIDAR_TC_VERIFY);
    launch_pdl(verify_select_kernel, n_seqs, 32, 0, c->stream, c->d_arg_idx, mix.n ? c->d_arg_idx + R : (const int32_t *)nullptr, c->d_step_seqs,
               c->d_forced, k, n_blocks, lay, cf.k_max, c->d_block, c->d_blk_len, c->d_step_n, c->d_step_L, c->d_seq_len, io, l.tl);
  }
  if (cf.debug & 2) {
    Launch l(c, TIDAR_TC_VERIFY);
    launch_pdl(kv_poison_kernel, dim3(n_seqs, cf.n_layers), 128, 0, c->stream, c->d_step_seqs, c->d_step_n, c->d_step_L, k, lay.k, geom(c), c->kv,
               c->pool_stride, l.tl);
  }
  CUDA_TRY(c, cudaGetLastError());
  return TIDAR_OK;
}

bool use_graphs(const tidar_ctx *c) { return c->cfg.impl == 0 && (c->graphs_ok || c->side_capture) && !c->timing && !(c->cfg.debug & (1 | 8)); }

void drop_graphs(tidar_ctx *c, size_t keep) {
  while (c->graphs.size() > keep) {
    cudaStreamSynchronize(c->stream);               // it may still be running
    cudaGraphExecDestroy(c->graphs.back().exec);
    c->graphs.pop_back();
  }
}

// Captures the step of `key` on stream st and keeps it as the most recently used graph.
bool capture_step(tidar_ctx *c, const tidar_ctx::StepKey &key, cudaStream_t st) {
  drop_graphs(c, tidar_ctx::MAX_GRAPHS - 1);
  tidar_ctx::StepGraph sg;
  sg.key = key;
  const int64_t l0 = c->launches;
  const cudaStream_t own = c->stream;
  cudaGraph_t graph = nullptr;
  int rc = TIDAR_OK;
  c->stream = st;
  cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    rc = record_step(c, key);
    e = cudaStreamEndCapture(st, &graph);
  }
  c->stream = own;
  if (e == cudaSuccess && rc == TIDAR_OK && graph) e = cudaGraphInstantiate(&sg.exec, graph, 0);
  if (graph) cudaGraphDestroy(graph);
  if (key.timeline) sg.tl_cls = c->tl_cls;
  sg.launches = c->launches - l0;
  c->launches = l0;
  if (e != cudaSuccess || rc != TIDAR_OK || !sg.exec) {
    cudaGetLastError();
    return false;
  }
  c->graphs.push_front(sg);
  c->graphs_captured++;
  return true;
}

// Behind a step that was launched kernel by kernel on the legacy default stream, while it runs: captures its shape once it has been run often enough.
// A capture and its graph cost the host about 9 us per launch, hidden behind the running step only where that is long enough, and a replayed launch is 0.3 -
// 0.5 us faster: worth it after some 16 steps, so a shape that was run that often is expected to come back.  (Tiny model, 23
// launches: 119 -> 107 us per step, 0.2 ms for the capture; 1.5B-class autoregressive step of 8 rows, 259 launches: 1.52 -> 1.43 ms.)  Steps of mixed block lengths seldom
// meet the same shape again and stay as they are.
constexpr int GRAPH_AFTER = 16;
void capture_aside(tidar_ctx *c, const tidar_ctx::StepKey &key) {
  if (key.mixed_R > 0 || key.timeline || key.count_tiles) return;
  auto it = std::find_if(c->seen.begin(), c->seen.end(), [&](const std::pair<tidar_ctx::StepKey, int> &s) { return s.first == key; });
  std::pair<tidar_ctx::StepKey, int> entry(key, 0);
  if (it != c->seen.end()) { entry = *it; c->seen.erase(it); }
  if (++entry.second < GRAPH_AFTER) {
    c->seen.push_front(entry);
    if (c->seen.size() > 2 * tidar_ctx::MAX_GRAPHS) c->seen.pop_back();
    return;
  }
  if (!c->capture_stream && cudaStreamCreateWithFlags(&c->capture_stream, cudaStreamNonBlocking) != cudaSuccess) { cudaGetLastError(); c->capture_stream = nullptr; c->side_capture = false; return; }
  if (!capture_step(c, key, c->capture_stream)) c->side_capture = false;
}

// The step proper.  Every launch of a step has the same arguments from step to step (lengths, page tables, token
// blocks and, for a step of mixed block lengths, the row layout live in device memory), except
// for the grid sizes, so on a stream of the caller's the step is captured once per key and replayed.  On the legacy default
// stream, which cannot be captured, that begins with a shape's seventeenth step (capture_aside).  Per-launch timing and the debug read-backs use plain
// launches of the same kernels.  key.units: attention units per KV head.
int launch_step(tidar_ctx *c, tidar_ctx::StepKey key) {
  key.timeline = c->timeline; key.count_tiles = c->count_tiles;
  if (c->cfg.impl == 0) {
    c->split_keys = key.split; c->attn_cluster = key.cluster; c->mixed_units = key.units;
    const int T = key.ar ? 1 : key.k * (key.k + 1);
    note_route(c, attention_plan(c, key.mixed_R > 0 ? key.mixed_R : key.n_seqs * T, key.mixed_R > 0 ? 0 : T));
  }
  if (!use_graphs(c)) return record_step(c, key);
  auto it = std::find_if(c->graphs.begin(), c->graphs.end(), [&](const tidar_ctx::StepGraph &g) { return g.key == key; });
  if (it == c->graphs.end()) {
    if (!c->graphs_ok) {
      if (int rc = record_step(c, key)) return rc;
      capture_aside(c, key);
      return TIDAR_OK;
    }
    if (!capture_step(c, key, c->stream)) {           // capture is not available here: plain launches from now on
      c->graphs_ok = false;
      return record_step(c, key);
    }
  } else if (it != c->graphs.begin()) {
    const tidar_ctx::StepGraph sg = *it;
    c->graphs.erase(it);
    c->graphs.push_front(sg);
  }
  const tidar_ctx::StepGraph &sg = c->graphs.front();
  CUDA_TRY(c, cudaGraphLaunch(sg.exec, c->stream));
  c->launches += sg.launches;
  c->graphs_launched++;
  if (key.timeline) { c->tl_cls = sg.tl_cls; c->tl_n = (int)sg.tl_cls.size(); }      // (another step may have been recorded since)
  return TIDAR_OK;
}

// Whether one more step may be enqueued: always when none is in flight; behind a step in flight only when
// every acceptance length of both is forced (the host then knows the lengths without reading the device),
// both use one block length for all their sequences and nothing reads per-step diagnostics.
bool may_enqueue(tidar_ctx *c, bool all_forced, bool mixed) {
  if (c->inflight.empty()) return true;
  if (c->inflight.size() >= 2 || !all_forced || mixed || c->timing || c->timeline || (c->cfg.debug & (1 | 8))) return false;
  return c->inflight.front().counted && c->inflight.front().ks.empty();
}

// Book-keeping of an enqueued step.  With every length forced the host advances the sequences now.
void push_flight(tidar_ctx *c, const int32_t *seqs, int n_seqs, const int32_t *forced, int k, const int32_t *ks) {
  tidar_ctx::Flight f;
  f.seqs.assign(seqs, seqs + n_seqs);
  if (ks) f.ks.assign(ks, ks + n_seqs);
  f.k = k; f.turn = c->turn++;
  f.counted = forced != nullptr;
  for (int i = 0; i < n_seqs && f.counted; ++i) f.counted = forced[i] > 0;
  if (f.counted)
    for (int i = 0; i < n_seqs; ++i) { c->seqs[seqs[i]].n += forced[i]; c->seqs[seqs[i]].k = ks ? ks[i] : k; }
  c->inflight.push_back(std::move(f));
}

// k_step: block length of this step (0 = the one the sequences' last pass left, which must then be
// the same for all of them); ar: plain autoregressive step (k_step is 1).
int enqueue_step(tidar_ctx *c, const int32_t *seqs, int n_seqs, const int32_t *forced, bool need_forced, int k_step = 0, bool ar = false) {
  const tidar_config &cf = c->cfg;
  if (!seqs || n_seqs < 1 || n_seqs > cf.max_batch) return fail(c, TIDAR_EINVAL, "n_seqs must be in [1, max_batch]");
  {
    bool all_forced = forced != nullptr;
    for (int i = 0; i < n_seqs && all_forced; ++i) all_forced = forced[i] > 0;
    if (!may_enqueue(c, all_forced && need_forced, false))
      return fail(c, TIDAR_EINVAL, c->inflight.size() >= 2 ? "two steps are already in flight; call tidar_step_wait first"
                                                            : "a step is in flight; call tidar_step_wait first (a second step can only follow with forced lengths, "
                                                              "one block length per step and no per-step diagnostics)");
  }
  if (k_step < 0 || k_step > cf.k_max) return fail(c, TIDAR_EINVAL, "block length %d outside [1, k_max = %d]", k_step, cf.k_max);
  int k = ar ? 1 : k_step;
  for (int i = 0; i < n_seqs; ++i) {
    const int q = seqs[i];
    if (q < 0 || q >= cf.max_batch || !c->seqs[q].active) return fail(c, TIDAR_EINVAL, "sequence %d is not prefilled", q);
    for (int j = 0; j < i; ++j) if (seqs[j] == q) return fail(c, TIDAR_EINVAL, "sequence %d listed twice", q);
    if (k == 0) k = c->seqs[q].k;
    else if (k_step == 0 && !ar && c->seqs[q].k != k)
      return fail(c, TIDAR_EINVAL, "the listed sequences hold blocks of different lengths; name the step's block length (tidar_step_k)");
    const int f = forced ? forced[i] : 0;
    if (f < 0 || f > k) return fail(c, TIDAR_EINVAL, "forced acceptance %d outside [0, %d]", f, k);
    if (need_forced && f == 0) return fail(c, TIDAR_EINVAL, "tidar_step_async needs a forced acceptance length per sequence");
    if (c->seqs[q].n + (ar ? 1 : 2 * k) > cf.max_seq_len)
      return fail(c, TIDAR_ECAPACITY, "sequence %d: n + %s = %d exceeds max_seq_len %d", q, ar ? "1" : "2k", c->seqs[q].n + (ar ? 1 : 2 * k), cf.max_seq_len);
  }
  for (int i = 0; i < n_seqs; ++i) {
    int rc = ensure_pages(c, seqs[i], c->seqs[seqs[i]].n + k);
    if (rc) return rc;
  }
  const int T = ar ? 1 : k * (k + 1), R = n_seqs * T;
  const int slot = c->turn & 1;
  for (int i = 0; i < n_seqs; ++i) {
    c->h_stage2[slot][i] = seqs[i]; c->h_stage2[slot][cf.max_batch + i] = forced ? forced[i] : 0;
    c->step_n[i] = c->seqs[seqs[i]].n;
  }
  const int spt = 2 * (128 / (cf.n_q_heads / cf.n_kv_heads));      // slots per attention unit (two query tiles)
  tidar_ctx::StepKey key;
  key.k = k; key.n_seqs = n_seqs; key.ar = ar; key.units = n_seqs * ((T + spt - 1) / spt);
  const StepAttention att = step_attention(c, c->step_n.data(), nullptr, k, n_seqs, ar, false);
  key.split = att.split; key.cluster = att.cluster;
  if (int rc = launch_step(c, key)) return rc;
  CUDA_TRY(c, cudaEventRecord(c->flight_done[slot], c->stream));
  push_flight(c, seqs, n_seqs, forced, k, nullptr);
  c->last_hidden_off = 0;
  c->last_rows = R + ((cf.beta < 1.0f && !ar) ? n_seqs * k : 0); c->last_first_pos = -1;      // the mixed rows follow the slots
  // the host tracks lengths without reading the device when L is forced
  return TIDAR_OK;
}

// A step in which listed sequence i uses block length ks[i] (Section 5: the block length follows the
// compute profile; nothing in the method ties the sequences of a batch to one length).  Equal lengths
// take the ordinary path; different lengths run over R = sum k_i (k_i + 1) rows with a per-sequence
// row layout and an attention unit table (one captured graph serves every step with the same
// number of sequences, row blocks of 16 and units).
int enqueue_step_mixed(tidar_ctx *c, const int32_t *seqs, int n_seqs, const int32_t *ks, const int32_t *forced) {
  const tidar_config &cf = c->cfg;
  if (!seqs || !ks || n_seqs < 1 || n_seqs > cf.max_batch) return fail(c, TIDAR_EINVAL, "n_seqs must be in [1, max_batch]");
  bool same = true;
  for (int i = 0; i < n_seqs; ++i) {
    if (ks[i] < 1 || ks[i] > cf.k_max) return fail(c, TIDAR_EINVAL, "block length %d of entry %d outside [1, k_max = %d]", ks[i], i, cf.k_max);
    same = same && ks[i] == ks[0];
  }
  if (same) return enqueue_step(c, seqs, n_seqs, forced, false, ks[0], false);
  if (!c->inflight.empty()) return fail(c, TIDAR_EINVAL, "a step is in flight; call tidar_step_wait first");
  for (int i = 0; i < n_seqs; ++i) {
    const int q = seqs[i], k = ks[i];
    if (q < 0 || q >= cf.max_batch || !c->seqs[q].active) return fail(c, TIDAR_EINVAL, "sequence %d is not prefilled", q);
    for (int j = 0; j < i; ++j) if (seqs[j] == q) return fail(c, TIDAR_EINVAL, "sequence %d listed twice", q);
    const int f = forced ? forced[i] : 0;
    if (f < 0 || f > k) return fail(c, TIDAR_EINVAL, "forced acceptance %d outside [0, %d]", f, k);
    if (c->seqs[q].n + 2 * k > cf.max_seq_len)
      return fail(c, TIDAR_ECAPACITY, "sequence %d: n + 2k = %d exceeds max_seq_len %d", q, c->seqs[q].n + 2 * k, cf.max_seq_len);
  }
  for (int i = 0; i < n_seqs; ++i)
    if (int rc = ensure_pages(c, seqs[i], c->seqs[seqs[i]].n + ks[i])) return rc;
  const int mb = cf.max_batch, spt = 2 * (128 / (cf.n_q_heads / cf.n_kv_heads));
  int32_t *hk = c->h_lay, *hoff = hk + (mb + 1), *hloc = hoff + (mb + 1), *ht0 = hloc + (mb + 1), *hte = ht0 + (c->R_head + mb);
  const int slot = c->turn & 1;
  int R = 0, loc = 0, tiles = 0, sum_k = 0;
  for (int i = 0; i < n_seqs; ++i) {
    const int k = ks[i], T = k * (k + 1);
    hk[i] = k; hoff[i] = R; hloc[i] = loc; sum_k += k;
    for (int r0 = R; r0 < R + T; r0 += spt) { ht0[tiles] = r0; hte[tiles] = R + T; ++tiles; }
    R += T; loc += k * k;
    c->h_stage2[slot][i] = seqs[i]; c->h_stage2[slot][mb + i] = forced ? forced[i] : 0;
    c->step_n[i] = c->seqs[seqs[i]].n;
  }
  hk[n_seqs] = 0; hoff[n_seqs] = R; hloc[n_seqs] = loc;
  // a mixed step's kernels take every per-sequence length from the staged layout: the nominal k is unused
  tidar_ctx::StepKey key;
  key.n_seqs = n_seqs; key.mixed_R = R; key.units = tiles;
  const StepAttention att = step_attention(c, c->step_n.data(), ks, 0, n_seqs, false, true);
  key.split = att.split; key.cluster = att.cluster;
  const int mixed_rows = cf.beta < 1.0f ? sum_k : 0;         // one mixed LM-head input row per verified position
  key.mixed_K = mixed_rows;
  // Steps of nearly the same size share one captured graph: rows are filled up to a multiple of 16 (the projections' row
  // blocks are that anyway) and units to a multiple of 4 with ones that have no rows.  (Also under debug bit 3, so that it differs in
  // the launch mode alone.)
  if (cf.impl == 0 && mixed_rows == 0 && c->graphs_ok) {
    key.mixed_R = (R + 15) / 16 * 16;
    for (; tiles % 4 && tiles < c->R_head + mb; ++tiles) ht0[tiles] = hte[tiles] = 0;
    key.units = tiles;
  }
  if (int rc = launch_step(c, key)) return rc;
  CUDA_TRY(c, cudaEventRecord(c->flight_done[slot], c->stream));
  push_flight(c, seqs, n_seqs, forced, 0, ks);
  c->last_hidden_off = 0;
  c->last_rows = R + mixed_rows; c->last_first_pos = -1;
  return TIDAR_OK;
}

// Waits for the oldest step in flight and hands out its results.
int finish_step(tidar_ctx *c, int32_t *out_tokens, int32_t *out_n) {
  if (c->inflight.empty()) return fail(c, TIDAR_EINVAL, "no step in flight");
  tidar_ctx::Flight f = std::move(c->inflight.front());
  c->inflight.pop_front();
  const int slot = f.turn & 1;
  // Everything up to the step is complete when this returns, as the caller is promised (the results, which the step's last kernel writes to
  // pinned memory, arrive a moment earlier).
  CUDA_TRY(c, cudaEventSynchronize(c->flight_done[slot]));
  const int32_t *done = c->h_done2[slot];
  if (done[0] != f.turn + 1) return fail(c, TIDAR_ECUDA, "the step's kernels ended without results");
  if (c->timing) collect_timing(c);
  if (c->timeline) collect_timeline(c);
  if (done[1]) {
    // The step's kernels have already rewritten the device-side lengths and blocks of the listed
    // sequences from invalid results: their state is lost, and so is that of a step enqueued behind
    // it.  Release them all; a new first pass is needed.
    const int st = done[1];
    cudaStreamSynchronize(c->stream);
    cudaMemsetAsync(c->d_status, 0, sizeof(int), c->stream);
    for (int q : f.seqs) release_sequence(c, q);
    for (auto &g : c->inflight) for (int q : g.seqs) release_sequence(c, q);
    c->inflight.clear();
    return fail(c, TIDAR_EDEVICE_TIMEOUT, "a bounded device-side wait gave up during the step (status %d); its results are invalid and the "
                                          "listed sequences were released (prefill them again)", st);
  }
  const int km = c->cfg.k_max;
  const int32_t *res = c->h_out2[slot];
  for (size_t i = 0; i < f.seqs.size(); ++i) {
    const int L = res[i * (km + 1)];
    if (!f.counted) {
      c->seqs[f.seqs[i]].n += L;
      c->seqs[f.seqs[i]].k = f.ks.empty() ? f.k : f.ks[i];        // entries of the block the step left
    }
    if (out_n) out_n[i] = L;
    if (out_tokens) for (int j = 0; j < km; ++j) out_tokens[i * km + j] = j < L ? res[i * (km + 1) + 1 + j] : -1;
  }
  return TIDAR_OK;
}

}  // namespace

// =============================================================================
extern "C" {

int tidar_arena_bytes(const tidar_config *cfg, size_t *out_bytes) {
  if (!cfg || !out_bytes) return fail(nullptr, TIDAR_EINVAL, "null argument");
  std::string why;
  if (int rc = validate(*cfg, why)) return fail(nullptr, rc, "%s", why.c_str());
  tidar_ctx tmp; tmp.cfg = *cfg;
  layout(tmp, nullptr, out_bytes);
  return TIDAR_OK;
}

int tidar_init(const tidar_config *cfg, const tidar_weights *w, void *arena, size_t arena_bytes, void *cuda_stream,
               tidar_ctx **out) {
  if (!cfg || !w || !arena || !out) return fail(nullptr, TIDAR_EINVAL, "null argument");
  std::string why;
  if (int rc = validate(*cfg, why)) return fail(nullptr, rc, "%s", why.c_str());
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) return fail(nullptr, TIDAR_ECUDA, "no CUDA device: this library has no CPU path");
  if (!w->embed || !w->lm_head || !w->final_norm || !w->attn_norm || !w->wqkv || !w->wo || !w->ffn_norm || !w->w_gate_up || !w->w_down)
    return fail(nullptr, TIDAR_EINVAL, "null weight pointer");
  if ((uintptr_t)arena % 256) return fail(nullptr, TIDAR_EINVAL, "arena must be 256-byte aligned");
  tidar_ctx *c = new tidar_ctx;
  c->cfg = *cfg;
  c->slab_bf16 = (cfg->debug & 4) != 0;
  c->stream = (cudaStream_t)cuda_stream;
  c->graphs_ok = c->stream != nullptr && c->stream != cudaStreamLegacy;
  c->side_capture = !c->graphs_ok && cfg->impl == 0;
  size_t need = 0;
  layout(*c, arena, &need);
  if (need > arena_bytes) { delete c; return fail(nullptr, TIDAR_ENOMEM, "arena has %zu bytes, %zu needed", arena_bytes, need); }
  c->embed = (const bf16 *)w->embed; c->lm_head = (const bf16 *)w->lm_head; c->final_norm = (const bf16 *)w->final_norm;
  for (int l = 0; l < cfg->n_layers; ++l) {
    if (!w->attn_norm[l] || !w->wqkv[l] || !w->wo[l] || !w->ffn_norm[l] || !w->w_gate_up[l] || !w->w_down[l]) {
      delete c; return fail(nullptr, TIDAR_EINVAL, "null weight pointer in layer %d", l);
    }
    c->attn_norm.push_back((const bf16 *)w->attn_norm[l]); c->wqkv.push_back((const bf16 *)w->wqkv[l]);
    c->wo.push_back((const bf16 *)w->wo[l]); c->ffn_norm.push_back((const bf16 *)w->ffn_norm[l]);
    c->wgu.push_back((const bf16 *)w->w_gate_up[l]); c->wdown.push_back((const bf16 *)w->w_down[l]);
  }
  if ((w->q_norm != nullptr) != (w->k_norm != nullptr)) { delete c; return fail(nullptr, TIDAR_EINVAL, "q_norm and k_norm come together or not at all"); }
  for (int l = 0; l < cfg->n_layers; ++l) {
    if (w->bqkv) { if (!w->bqkv[l]) { delete c; return fail(nullptr, TIDAR_EINVAL, "null bqkv pointer in layer %d", l); } c->bqkv.push_back((const bf16 *)w->bqkv[l]); }
    if (w->q_norm) {
      if (!w->q_norm[l] || !w->k_norm[l]) { delete c; return fail(nullptr, TIDAR_EINVAL, "null q_norm / k_norm pointer in layer %d", l); }
      c->q_norm.push_back((const bf16 *)w->q_norm[l]); c->k_norm.push_back((const bf16 *)w->k_norm[l]);
    }
  }
  if (cfg->impl == 0) {
    if (int rc = init_tensor_core_path(c)) { std::string m = c->err; delete c; return fail(nullptr, rc, "%s", m.c_str()); }
  }
  c->seqs.resize(cfg->max_batch);
  c->step_n.resize(cfg->max_batch);
  // free list in a scrambled order so that page tables are never contiguous
  c->free_pages.resize(c->n_pages);
  for (int i = 0; i < c->n_pages; ++i) c->free_pages[i] = i;
  uint32_t st = 0x9e3779b9u;
  for (int i = c->n_pages - 1; i > 0; --i) { st = st * 1664525u + 1013904223u; std::swap(c->free_pages[i], c->free_pages[(st >> 8) % (i + 1)]); }
  // one pinned block: first-pass result | per slot: step results, staged inputs, turn and status | mixed-step layout | page-table mirror
  const size_t n_out = (size_t)cfg->max_batch * (cfg->k_max + 1), n_stage = 2 * (size_t)cfg->max_batch, n_pt = (size_t)cfg->max_batch * c->pages_per_seq;
  cudaError_t e = cudaHostAlloc((void **)&c->h_pinned, (n_out + 2 * (n_out + n_stage + 16) + c->lay_ints + n_pt) * sizeof(int), cudaHostAllocDefault);
  if (e != cudaSuccess) { delete c; return fail(nullptr, TIDAR_ECUDA, "cudaHostAlloc: %s", cudaGetErrorString(e)); }
  {
    int32_t *p = c->h_pinned + n_out;
    for (int sl = 0; sl < 2; ++sl) {
      c->h_out2[sl] = p; p += n_out;
      c->h_stage2[sl] = p; p += n_stage;
      c->h_done2[sl] = p; p += 16;
      c->h_done2[sl][0] = c->h_done2[sl][1] = 0;
    }
    c->h_lay = p; p += c->lay_ints;
    c->h_page_table = p;
    std::memset(c->h_page_table, 0, n_pt * sizeof(int));
  }
  e = cudaMemsetAsync(c->d_seq_len, 0, cfg->max_batch * sizeof(int), c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->d_status, 0, 64 * sizeof(int), c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->d_page_table, 0, (size_t)cfg->max_batch * c->pages_per_seq * sizeof(int), c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) { cudaFreeHost(c->h_pinned); delete c; return fail(nullptr, TIDAR_ECUDA, "arena set-up: %s", cudaGetErrorString(e)); }
  for (cudaEvent_t &ev : c->flight_done)
    if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) {
      if (c->flight_done[0]) cudaEventDestroy(c->flight_done[0]);
      cudaFreeHost(c->h_pinned); delete c; return fail(nullptr, TIDAR_ECUDA, "cudaEventCreate failed");
    }
  *out = c;
  return TIDAR_OK;
}

int tidar_prefill(tidar_ctx *c, int32_t seq, const int32_t *prompt, int32_t n_prompt, int32_t k, int32_t *out_first) {
  if (!c) return TIDAR_EINVAL;
  const tidar_config &cf = c->cfg;
  if (!c->inflight.empty()) return fail(c, TIDAR_EINVAL, "a step is in flight");
  if (seq < 0 || seq >= cf.max_batch) return fail(c, TIDAR_EINVAL, "seq %d out of range", seq);
  if (!prompt || n_prompt < 1) return fail(c, TIDAR_EINVAL, "empty prompt");
  if (k < 1 || k > cf.k_max) return fail(c, TIDAR_EINVAL, "k must be in [1, k_max]");
  if (n_prompt + 2 * k > cf.max_seq_len) return fail(c, TIDAR_ECAPACITY, "n_prompt + 2k = %d exceeds max_seq_len %d", n_prompt + 2 * k, cf.max_seq_len);
  for (int i = 0; i < n_prompt; ++i)
    if (prompt[i] < 0 || prompt[i] >= cf.vocab) return fail(c, TIDAR_EINVAL, "prompt id %d at %d out of range", prompt[i], i);
  SeqState &s = c->seqs[seq];
  release_sequence(c, seq);
  s.k = k;
  if (int rc = ensure_pages(c, seq, n_prompt + k)) return rc;
  CUDA_TRY(c, cudaMemcpyAsync(c->d_prompt, prompt, (size_t)n_prompt * sizeof(int), cudaMemcpyHostToDevice, c->stream));
  const int total = n_prompt + k;
  const int last_rows = std::min(total, c->R_cap - (cf.beta < 1.0f ? 1 : 0));     // the last chunk may carry one mixed row
  int row0 = 0;
  while (row0 < total) {
    const bool last = row0 >= total - last_rows;
    const int rows = last ? total - row0 : std::min(c->R_cap, total - last_rows - row0);
    {
      Launch l(c, TIDAR_TC_EMBED);
      assemble_prefill_kernel<<<rows, 256, 0, c->stream>>>(c->meta, seq, row0, n_prompt, k, cf.mask_token_id, c->d_prompt, c->embed,
                                                           cf.d_model, c->X, cf.temperature > 0.f ? 1 : 0, (unsigned long long)cf.sample_seed);
    }
    // beta < 1: the settled first token mixes the last prompt row with the first mask row
    MixRows mix;
    const int rlp = n_prompt - 1 - row0;               // the last prompt row inside this chunk
    if (last && cf.beta < 1.0f) { mix.n = 1; mix.k = 1; mix.a0 = rlp; mix.b0 = rlp + 1; }
    // logits are needed for the last prompt row and the k mask rows only; the LM head runs on the
    // trailing rows of the last chunk, as many as a decode step has (all of them for a short prompt)
    c->split_keys = may_split(row0 + rows); c->attn_cluster = 1;
    const int head_row0 = last ? std::max(0, rows + mix.n - c->R_head) : 0;
    if (int rc = forward_rows(c, rows, last, rows, mix, head_row0)) return rc;
    if (last) {
      Launch l(c, TIDAR_TC_VERIFY);
      prefill_finish_kernel<<<1, 32, 0, c->stream>>>(c->d_arg_idx, rlp - head_row0, (mix.n ? rows : rlp) - head_row0, k, cf.k_max, seq, n_prompt,
                                                     c->d_block, c->d_blk_len, c->d_seq_len, c->d_status, c->h_pinned);
      c->last_rows = rows - head_row0; c->last_first_pos = row0 + head_row0; c->last_hidden_off = head_row0;
    }
    row0 += rows;
  }
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  if (c->timing) collect_timing(c);
  if (const int st = c->h_pinned[1]) {
    cudaMemsetAsync(c->d_status, 0, sizeof(int), c->stream);
    release_sequence(c, seq);
    return device_timeout(c, st);
  }
  s.n = n_prompt; s.active = true;
  if (out_first) *out_first = c->h_pinned[0];
  return TIDAR_OK;
}

int tidar_step(tidar_ctx *c, const int32_t *seqs, int32_t n_seqs, const int32_t *forced, int32_t *out_tokens, int32_t *out_n) {
  if (!c) return TIDAR_EINVAL;
  if (int rc = enqueue_step(c, seqs, n_seqs, forced, false)) return rc;
  return finish_step(c, out_tokens, out_n);
}

int tidar_step_async(tidar_ctx *c, const int32_t *seqs, int32_t n_seqs, const int32_t *forced) {
  if (!c) return TIDAR_EINVAL;
  if (!forced) return fail(c, TIDAR_EINVAL, "tidar_step_async needs forced acceptance lengths");
  return enqueue_step(c, seqs, n_seqs, forced, true);
}

int tidar_step_wait(tidar_ctx *c, int32_t *out_tokens, int32_t *out_n) {
  if (!c) return TIDAR_EINVAL;
  return finish_step(c, out_tokens, out_n);
}

int tidar_step_k(tidar_ctx *c, const int32_t *seqs, int32_t n_seqs, int32_t k, const int32_t *forced, int32_t *out_tokens, int32_t *out_n) {
  if (!c) return TIDAR_EINVAL;
  if (k < 1) return fail(c, TIDAR_EINVAL, "block length must be at least 1");
  if (int rc = enqueue_step(c, seqs, n_seqs, forced, false, k, false)) return rc;
  return finish_step(c, out_tokens, out_n);
}

int tidar_step_ks(tidar_ctx *c, const int32_t *seqs, int32_t n_seqs, const int32_t *ks, const int32_t *forced, int32_t *out_tokens, int32_t *out_n) {
  if (!c) return TIDAR_EINVAL;
  if (int rc = enqueue_step_mixed(c, seqs, n_seqs, ks, forced)) return rc;
  return finish_step(c, out_tokens, out_n);
}

int tidar_ar_step(tidar_ctx *c, const int32_t *seqs, int32_t n_seqs, int32_t *out_tokens) {
  if (!c) return TIDAR_EINVAL;
  if (int rc = enqueue_step(c, seqs, n_seqs, nullptr, false, 1, true)) return rc;
  std::vector<int32_t> toks((size_t)std::max(n_seqs, 1) * c->cfg.k_max), ls(std::max(n_seqs, 1));
  if (int rc = finish_step(c, toks.data(), ls.data())) return rc;
  if (out_tokens) for (int i = 0; i < n_seqs; ++i) out_tokens[i] = toks[(size_t)i * c->cfg.k_max];
  return TIDAR_OK;
}

int tidar_ridge_k(const tidar_ctx *c, int32_t n_seqs, int32_t row_budget) {
  if (!c || n_seqs < 1) return TIDAR_EINVAL;
  if (row_budget <= 0) row_budget = 288;       // one row block of the projections: where the 8B-class step turns tensor-bound
  int k = 1;
  while (k < c->cfg.k_max && (long long)n_seqs * (k + 1) * (k + 2) <= row_budget) ++k;
  return k;
}

int tidar_plan_ks(int32_t n_seqs, int32_t k_max, int32_t row_budget, const int32_t *want, int32_t *out_ks) {
  if (n_seqs < 1 || k_max < 1 || !out_ks) return fail(nullptr, TIDAR_EINVAL, "tidar_plan_ks: n_seqs and k_max must be positive, out_ks non-null");
  if (row_budget <= 0) row_budget = 288;
  long long rows = 0;
  for (int i = 0; i < n_seqs; ++i) {
    if (want && want[i] < 1) return fail(nullptr, TIDAR_EINVAL, "tidar_plan_ks: want[%d] = %d, must be at least 1", i, want[i]);
    out_ks[i] = 1; rows += 2;
  }
  // One more draft for a sequence at length k costs 2(k + 1) rows and can yield one more token: the cost
  // grows with k, so the shortest block that may still grow is always the best place for the next rows.
  for (;;) {
    int best = -1;
    for (int i = 0; i < n_seqs; ++i) {
      const int cap = want ? std::min(k_max, want[i]) : k_max;
      if (out_ks[i] < cap && (best < 0 || out_ks[i] < out_ks[best])) best = i;
    }
    if (best < 0 || rows + 2 * (out_ks[best] + 1) > row_budget) break;
    rows += 2 * (out_ks[best] + 1);
    out_ks[best]++;
  }
  return TIDAR_OK;
}

int tidar_release(tidar_ctx *c, int32_t seq) {
  if (!c) return TIDAR_EINVAL;
  if (!c->inflight.empty()) return fail(c, TIDAR_EINVAL, "a step is in flight");
  if (seq < 0 || seq >= c->cfg.max_batch) return fail(c, TIDAR_EINVAL, "seq %d out of range", seq);
  if (c->seqs[seq].active) release_sequence(c, seq);
  return TIDAR_OK;
}

int tidar_score(tidar_ctx *c, int32_t seq, const int32_t *ids, int32_t n, float *logprobs) {
  if (!c) return TIDAR_EINVAL;
  const tidar_config &cf = c->cfg;
  if (!c->inflight.empty()) return fail(c, TIDAR_EINVAL, "a step is in flight");
  if (seq < 0 || seq >= cf.max_batch) return fail(c, TIDAR_EINVAL, "seq %d out of range", seq);
  if (!ids || !logprobs || n < 2) return fail(c, TIDAR_EINVAL, "tidar_score needs at least two token ids");
  if (n > cf.max_seq_len) return fail(c, TIDAR_ECAPACITY, "%d tokens exceed max_seq_len %d", n, cf.max_seq_len);
  for (int i = 0; i < n; ++i)
    if (ids[i] < 0 || ids[i] >= cf.vocab) return fail(c, TIDAR_EINVAL, "token id %d at %d out of range", ids[i], i);
  release_sequence(c, seq);
  c->seqs[seq].k = 1;
  if (int rc = ensure_pages(c, seq, n)) return rc;
  CUDA_TRY(c, cudaMemcpyAsync(c->d_prompt, ids, (size_t)n * sizeof(int), cudaMemcpyHostToDevice, c->stream));
  const int d = cf.d_model;
  for (int row0 = 0; row0 < n - 1; row0 += c->R_cap) {
    const int rows = std::min(c->R_cap, n - 1 - row0);          // the last token predicts nothing that is scored
    {
      Launch l(c, TIDAR_TC_EMBED);
      assemble_prefill_kernel<<<rows, 256, 0, c->stream>>>(c->meta, seq, row0, n, 0, cf.mask_token_id, c->d_prompt, c->embed, d, c->X, 0, 0ull);
    }
    c->split_keys = may_split(row0 + rows); c->attn_cluster = 1;
    if (int rc = forward_rows(c, rows, false, rows)) return rc;      // ends with the final norm in c->A
    const int32_t *target = c->d_prompt + row0 + 1;
    if (cf.impl == 0) {
      // (Through fp32 logits in 16384-id chunks, each reduced by a kernel of its own, 1776 rows of a 1536-wide 152 k vocabulary took 1.39 ms;
      // this way 0.63, 1.3 PFLOP/s.)
      if (int rc = gemm_tc_launch(c, gemm_tc::MODE_LSE, c->A, c->R_cap, c->tm_lm, rows, cf.vocab, d, TIDAR_TC_LMHEAD, nullptr, nullptr, nullptr, 0, nullptr, target)) return rc;
      Launch ll(c, TIDAR_TC_LMHEAD);
      launch_pdl(score_merge_kernel, (rows + 15) / 16, 512, 0, c->stream, (const float2 *)c->partials, gemm_tc::lse_parts(cf.vocab), c->d_tgt_logit, rows, c->d_logprob);
    } else {
      for (int v0 = 0; v0 < cf.vocab; v0 += c->lm_chunk) {
        const int nc = std::min(c->lm_chunk, cf.vocab - v0);
        int S = 1; size_t stride = 0;
        if (int rc = gemm_partials(c, c->A, c->R_cap, c->lm_head + (size_t)v0 * d, nullptr, rows, nc, d, c->partials, &S, &stride, TIDAR_TC_LMHEAD)) return rc;
        Launch ll(c, TIDAR_TC_LMHEAD);
        score_chunk_kernel<<<rows, 256, 0, c->stream>>>(c->partials, nc, nc, v0, v0 == 0, target, c->d_run_max, c->d_run_sum, c->d_tgt_logit);
      }
      Launch ll(c, TIDAR_TC_LMHEAD);
      score_finish_kernel<<<(rows + 127) / 128, 128, 0, c->stream>>>(c->d_run_max, c->d_run_sum, c->d_tgt_logit, rows, c->d_logprob);
    }
    CUDA_TRY(c, cudaMemcpyAsync(logprobs + row0, c->d_logprob, (size_t)rows * sizeof(float), cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  }
  CUDA_TRY(c, cudaGetLastError());
  if (c->timing) collect_timing(c);
  release_sequence(c, seq);                         // the slot was scratch for this call
  return check_device_status(c);
}

int tidar_free(tidar_ctx *c) {
  if (!c) return TIDAR_EINVAL;
  cudaStreamSynchronize(c->stream);
  for (auto &t : c->timed) { cudaEventDestroy(t.a); cudaEventDestroy(t.b); }
  drop_graphs(c, 0);
  if (c->capture_stream) cudaStreamDestroy(c->capture_stream);
  for (cudaEvent_t ev : c->flight_done) cudaEventDestroy(ev);
  if (c->h_pinned) cudaFreeHost(c->h_pinned);
  delete c;
  return TIDAR_OK;
}

const char *tidar_last_error(const tidar_ctx *c) { return c ? c->err.c_str() : g_init_error.c_str(); }

int tidar_seq_len(const tidar_ctx *c, int32_t seq) {
  if (!c || seq < 0 || seq >= c->cfg.max_batch || !c->seqs[seq].active) return TIDAR_EINVAL;
  return c->seqs[seq].n;
}

int64_t tidar_launch_count(const tidar_ctx *c) { return c ? c->launches : -1; }

int tidar_debug_set_block(tidar_ctx *c, int32_t seq, const int32_t *block) {
  if (!c || !block) return TIDAR_EINVAL;
  if (seq < 0 || seq >= c->cfg.max_batch || !c->seqs[seq].active) return fail(c, TIDAR_EINVAL, "sequence %d is not prefilled", seq);
  CUDA_TRY(c, cudaMemcpyAsync(c->d_block + (size_t)seq * c->cfg.k_max, block, c->seqs[seq].k * sizeof(int), cudaMemcpyHostToDevice, c->stream));
  CUDA_TRY(c, cudaMemcpyAsync(c->d_blk_len + seq, &c->seqs[seq].k, sizeof(int), cudaMemcpyHostToDevice, c->stream));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return TIDAR_OK;
}

int tidar_debug_get_block(tidar_ctx *c, int32_t seq, int32_t *block) {
  if (!c || !block) return TIDAR_EINVAL;
  if (seq < 0 || seq >= c->cfg.max_batch || !c->seqs[seq].active) return fail(c, TIDAR_EINVAL, "sequence %d is not prefilled", seq);
  CUDA_TRY(c, cudaMemcpyAsync(block, c->d_block + (size_t)seq * c->cfg.k_max, c->seqs[seq].k * sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return TIDAR_OK;
}

int tidar_debug_last_rows(const tidar_ctx *c, int32_t *n_rows, int32_t *first_pos) {
  if (!c) return TIDAR_EINVAL;
  if (n_rows) *n_rows = c->last_rows;
  if (first_pos) *first_pos = c->last_first_pos;
  return TIDAR_OK;
}

static int check_rows(tidar_ctx *c, int row0, int n) {
  if (row0 < 0 || n < 1 || row0 + n > c->last_rows) return fail(c, TIDAR_EINVAL, "rows [%d, %d) outside the last pass (%d rows)", row0, row0 + n, c->last_rows);
  return TIDAR_OK;
}

int tidar_debug_get_logits(tidar_ctx *c, int32_t row0, int32_t n, float *out) {
  if (!c || !out) return TIDAR_EINVAL;
  if (!c->dbg_logits) return fail(c, TIDAR_EINVAL, "context was created without debug bit 0");
  if (int rc = check_rows(c, row0, n)) return rc;
  CUDA_TRY(c, cudaMemcpyAsync(out, c->dbg_logits + (size_t)row0 * c->cfg.vocab, (size_t)n * c->cfg.vocab * sizeof(float), cudaMemcpyDeviceToHost, c->stream));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return TIDAR_OK;
}

int tidar_debug_get_hidden(tidar_ctx *c, int32_t layer, int32_t row0, int32_t n, float *out) {
  if (!c || !out) return TIDAR_EINVAL;
  if (!c->dbg_hidden) return fail(c, TIDAR_EINVAL, "context was created without debug bit 0");
  if (layer < 0 || layer > c->cfg.n_layers) return fail(c, TIDAR_EINVAL, "layer out of range");
  if (int rc = check_rows(c, row0, n)) return rc;
  const size_t d = c->cfg.d_model;
  CUDA_TRY(c, cudaMemcpyAsync(out, c->dbg_hidden + ((size_t)layer * c->R_cap + c->last_hidden_off + row0) * d, (size_t)n * d * sizeof(float),
                              cudaMemcpyDeviceToHost, c->stream));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return TIDAR_OK;
}

int tidar_debug_get_argmax(tidar_ctx *c, int32_t row0, int32_t n, int32_t *out) {
  if (!c || !out) return TIDAR_EINVAL;
  if (int rc = check_rows(c, row0, n)) return rc;
  CUDA_TRY(c, cudaMemcpyAsync(out, c->d_arg_idx + row0, (size_t)n * sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return TIDAR_OK;
}

int tidar_debug_get_kv(tidar_ctx *c, int32_t seq, int32_t layer, int32_t pos0, int32_t npos, uint16_t *k_out, uint16_t *v_out) {
  if (!c || !k_out || !v_out) return TIDAR_EINVAL;
  if (seq < 0 || seq >= c->cfg.max_batch || !c->seqs[seq].active) return fail(c, TIDAR_EINVAL, "sequence %d is not prefilled", seq);
  if (layer < 0 || layer >= c->cfg.n_layers) return fail(c, TIDAR_EINVAL, "layer out of range");
  const int backed = (int)c->seqs[seq].pages.size() * c->cfg.page_size;
  if (pos0 < 0 || npos < 1 || pos0 + npos > backed) return fail(c, TIDAR_EINVAL, "positions [%d, %d) not backed by pages (%d)", pos0, pos0 + npos, backed);
  const size_t per = (size_t)c->cfg.n_kv_heads * c->cfg.head_dim;
  const bf16 *Kp = c->kv + (size_t)(2 * layer) * c->pool_stride, *Vp = Kp + c->pool_stride;
  for (int p = 0; p < npos; p += 256) {
    const int np = std::min(256, npos - p);
    bf16 *ko = c->dbg_kv, *vo = c->dbg_kv + 256 * per;
    kv_gather_kernel<<<dim3(np, c->cfg.n_kv_heads), 64, 0, c->stream>>>(Kp, Vp, geom(c), seq, pos0 + p, ko, vo);
    CUDA_TRY(c, cudaMemcpyAsync(k_out + (size_t)p * per, ko, np * per * 2, cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaMemcpyAsync(v_out + (size_t)p * per, vo, np * per * 2, cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  }
  return TIDAR_OK;
}

int tidar_debug_wait_probe(tidar_ctx *c, int32_t limit_polls) {
  if (!c) return TIDAR_EINVAL;
  if (c->cfg.impl != 0) return fail(c, TIDAR_EINVAL, "the bounded waits exist in the tensor-core kernels only");
  if (limit_polls < 1 || limit_polls > (1 << 20)) return fail(c, TIDAR_EINVAL, "limit_polls must be in [1, 2^20]");
  wait_probe_kernel<<<1, 32, 0, c->stream>>>((uint32_t)limit_polls, c->d_status, c->d_status + 8);
  CUDA_TRY(c, cudaGetLastError());
  return TIDAR_OK;
}

int tidar_debug_force_status(tidar_ctx *c, int32_t value) {
  if (!c) return TIDAR_EINVAL;
  CUDA_TRY(c, cudaMemcpyAsync(c->d_status, &value, sizeof(int), cudaMemcpyHostToDevice, c->stream));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return TIDAR_OK;
}

int tidar_debug_count_attention_tiles(tidar_ctx *c, int32_t on, uint64_t *visited) {
  if (!c) return TIDAR_EINVAL;
  if (c->cfg.impl != 0) return fail(c, TIDAR_EINVAL, "the tile counter exists for the tensor-core attention kernel only");
  unsigned long long *ctr = c->d_tl + 2 * tidar_ctx::TL_MAX;
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  if (visited) {
    unsigned long long v = 0;
    CUDA_TRY(c, cudaMemcpy(&v, ctr, sizeof v, cudaMemcpyDeviceToHost));
    *visited = v;
  }
  CUDA_TRY(c, cudaMemset(ctr, 0, sizeof(unsigned long long)));
  c->count_tiles = on != 0;
  return TIDAR_OK;
}

int tidar_debug_set_timeline(tidar_ctx *c, int32_t on) {
  if (!c) return TIDAR_EINVAL;
  if (c->cfg.impl != 0) return fail(c, TIDAR_EINVAL, "the in-kernel timeline exists for the tensor-core kernels only");
  c->timeline = on != 0;
  return TIDAR_OK;
}

int tidar_debug_get_timeline(tidar_ctx *c, float *class_ms, float *busy_ms, float *span_ms) {
  if (!c || !class_ms) return TIDAR_EINVAL;
  for (int i = 0; i < TIDAR_TC_COUNT; ++i) class_ms[i] = c->tl_class_ms[i];
  if (busy_ms) *busy_ms = c->tl_busy_ms;
  if (span_ms) *span_ms = c->tl_span_ms;
  return TIDAR_OK;
}

int tidar_debug_graph_stats(const tidar_ctx *c, int64_t *captured, int64_t *launched, int32_t *kept) {
  if (!c) return TIDAR_EINVAL;
  if (captured) *captured = c->graphs_captured;
  if (launched) *launched = c->graphs_launched;
  if (kept) *kept = (int32_t)c->graphs.size();
  return TIDAR_OK;
}

int tidar_debug_attention_route(tidar_ctx *c, int32_t *out) {
  if (!c || !out) return TIDAR_EINVAL;
  if (c->cfg.impl != 0) return fail(c, TIDAR_EINVAL, "tensor-core path only");
  if (!c->inflight.empty()) return fail(c, TIDAR_EINVAL, "a step is in flight");
  out[0] = c->route.cluster; out[1] = c->route.merge ? 1 : 0; out[2] = -1;
  if (c->route.plan_units > 0) {
    std::vector<attn_tc::Tile> tiles(2 * (size_t)c->route.plan_units);
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    CUDA_TRY(c, cudaMemcpy(tiles.data(), c->plan_tiles, tiles.size() * sizeof(tiles[0]), cudaMemcpyDeviceToHost));
    out[2] = (int32_t)std::count_if(tiles.begin(), tiles.end(), [](const attn_tc::Tile &t) { return t.n_items > 1; });
  }
  return TIDAR_OK;
}

int tidar_debug_plan_projection(const tidar_config *cfg, int32_t n_sms, int32_t swiglu, int32_t R, int32_t N, int32_t K, int32_t *out) {
  std::string why;
  if (!cfg || !out) return fail(nullptr, TIDAR_EINVAL, "null argument");
  if (validate(*cfg, why) != TIDAR_OK) return fail(nullptr, TIDAR_EINVAL, "%s", why.c_str());
  if (n_sms < 2 || n_sms > MAX_SMS || R < 1 || N < 1 || K < 64) return fail(nullptr, TIDAR_EINVAL, "n_sms, R, N or K out of range");
  tidar_ctx c;
  size_t need = 0;
  c.cfg = *cfg; c.n_sms = n_sms;
  layout(c, nullptr, &need);
  const gemm_tc::Args a = plan_gemm(&c, swiglu ? gemm_tc::MODE_SWIGLU : gemm_tc::MODE_SLAB, R, N, K);
  out[0] = a.n_rb; out[1] = a.rb_rows; out[2] = a.S; out[3] = a.total_items(); out[4] = a.warm_epilogue;
  return TIDAR_OK;
}

int tidar_debug_plan_norm(int32_t n_sms, int32_t R, int32_t d, int32_t S, int32_t *out) {
  if (!out || n_sms < 1 || R < 1 || d < 1 || S < 0 || S > MAX_SLABS) return fail(nullptr, TIDAR_EINVAL, "argument out of range");
  const NormPlan p = norm_plan(n_sms, R, d, S, true);
  out[0] = p.bulk ? 1 : 0; out[1] = (int32_t)p.smem;
  return TIDAR_OK;
}

int tidar_debug_plan_step(const tidar_config *cfg, int32_t n_sms, const int32_t *max_clusters, const int32_t *n, const int32_t *ks, int32_t n_seqs, int32_t ar, int32_t *out) {
  std::string why;
  if (!cfg || !max_clusters || !n || !ks || !out) return fail(nullptr, TIDAR_EINVAL, "null argument");
  if (validate(*cfg, why) != TIDAR_OK) return fail(nullptr, TIDAR_EINVAL, "%s", why.c_str());
  if (n_sms < 1 || n_sms > MAX_SMS || n_seqs < 1) return fail(nullptr, TIDAR_EINVAL, "n_sms or n_seqs out of range");
  for (int i = 0; i < n_seqs; ++i) if (n[i] < 0 || ks[i] < 1 || ks[i] > cfg->k_max) return fail(nullptr, TIDAR_EINVAL, "length or block length %d out of range", i);
  tidar_ctx c;
  c.cfg = *cfg; c.n_sms = n_sms;
  for (int i = 0; i < 3; ++i) c.max_clusters[2 << i] = max_clusters[i];
  const bool mixed = std::any_of(ks, ks + n_seqs, [&](int k) { return k != ks[0]; });
  const StepAttention a = step_attention(&c, n, mixed ? ks : nullptr, ks[0], n_seqs, ar != 0, mixed);
  out[0] = a.cluster; out[1] = a.split ? 1 : 0;
  return TIDAR_OK;
}

int tidar_debug_set_timing(tidar_ctx *c, int32_t on) {
  if (!c) return TIDAR_EINVAL;
  c->timing = on != 0;
  return TIDAR_OK;
}

int tidar_debug_get_timing(tidar_ctx *c, float *ms) {
  if (!c || !ms) return TIDAR_EINVAL;
  for (int i = 0; i < TIDAR_TC_COUNT; ++i) ms[i] = c->class_ms[i];
  return TIDAR_OK;
}

int tidar_gemm(tidar_ctx *c, const void *A, const void *W, int32_t R, int32_t N, int32_t K, int32_t splits, float *out) {
  if (!c) return TIDAR_EINVAL;
  if (!A || !W || !out) return fail(c, TIDAR_EINVAL, "null argument");
  if (!c->inflight.empty()) return fail(c, TIDAR_EINVAL, "a step is in flight");
  if (R < 1 || N < 1 || K < 64 || K % 64) return fail(c, TIDAR_EINVAL, "R, N >= 1 and K a positive multiple of 64 required");
  if (((uintptr_t)A | (uintptr_t)W) % 16) return fail(c, TIDAR_EINVAL, "A and W must be 16-byte aligned");
  if (splits < 0 || splits > c->S_max) return fail(c, TIDAR_EINVAL, "splits must be in [0, %d]", c->S_max);
  const size_t need = (size_t)(splits > 0 ? splits : c->S_max) * R * N;
  if (need > c->partials_cap) return fail(c, TIDAR_ECAPACITY, "R*N*splits = %zu floats exceed the context's scratch (%zu)", need, c->partials_cap);
  int S = 1; size_t stride = 0;
  if (c->cfg.impl == 0) {
    tidar_ctx::WMap tmW;
    if (!encode_weights(c, &tmW, W, N, K))
      return fail(c, TIDAR_ECUDA, "cuTensorMapEncodeTiled failed for W");
    if (int rc = gemm_tc_launch(c, gemm_tc::MODE_SLAB, (const bf16 *)A, R, tmW, R, N, K, TIDAR_TC_GEMM, &S, &stride, c->partials, splits)) return rc;
  } else {
    if (int rc = gemm_partials(c, (const bf16 *)A, R, (const bf16 *)W, nullptr, R, N, K, c->partials, &S, &stride, TIDAR_TC_GEMM)) return rc;
  }
  {
    Launch l(c, TIDAR_TC_GEMM);
    const size_t n = (size_t)R * N;
    slab_sum_kernel<<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(c->partials, S, stride, n, out);
  }
  CUDA_TRY(c, cudaGetLastError());
  return TIDAR_OK;
}

int tidar_sync(tidar_ctx *c) {
  if (!c) return TIDAR_EINVAL;
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return check_device_status(c);
}

int tidar_attention(tidar_ctx *c, const void *q, const void *k_pages, const void *v_pages, int32_t n_pages, const int32_t *page_table,
                    int32_t pages_per_seq, const int32_t *seq_len, const void *k_local, const void *v_local, void *out,
                    int32_t n_seqs, int32_t k) {
  if (!c) return TIDAR_EINVAL;
  if (!q || !k_pages || !v_pages || !page_table || !seq_len || !k_local || !v_local || !out) return fail(c, TIDAR_EINVAL, "null argument");
  if (k < 1 || k > c->cfg.k_max || n_seqs < 1 || n_seqs * k * (k + 1) > c->R_cap) return fail(c, TIDAR_EINVAL, "n_seqs * k(k+1) exceeds the context's row capacity");
  if (n_pages < 1 || pages_per_seq < 1) return fail(c, TIDAR_EINVAL, "n_pages and pages_per_seq must be positive");
  if ((long long)pages_per_seq * c->cfg.page_size < k) return fail(c, TIDAR_EINVAL, "the page table cannot back the k causal slots");
  if (!c->inflight.empty()) return fail(c, TIDAR_EINVAL, "a step is in flight");
  if (((uintptr_t)q | (uintptr_t)k_pages | (uintptr_t)v_pages | (uintptr_t)k_local | (uintptr_t)v_local | (uintptr_t)out) % 16 ||
      ((uintptr_t)page_table | (uintptr_t)seq_len) % 4)
    return fail(c, TIDAR_EINVAL, "tensors must be 16-byte aligned (page_table and seq_len 4-byte)");
  const int R = n_seqs * k * (k + 1), n_max = pages_per_seq * c->cfg.page_size - k;
  const KvGeom g{c->cfg.n_kv_heads, c->cfg.head_dim, c->cfg.page_size, pages_per_seq, page_table, n_pages};
  if (c->cfg.impl == 0) {
    const DirectPlan d = attention_direct(c, n_seqs, k, pages_per_seq);
    attn_tc::PlanArgs plan{};
    if (!d.streams) {                              // (launched ahead of the host's work on the tensor maps)
      c->split_keys = may_split(pages_per_seq * c->cfg.page_size); c->attn_cluster = 1;       // the lengths themselves are on the device
      plan = attention_plan(c, R, k * (k + 1));
      note_route(c, plan);
      Launch l(c, TIDAR_TC_EMBED);
      launch_pdl(attn_meta_plan_kernel, 1 + (R + 511) / 512, 512, 0, c->stream, c->meta, seq_len, k, R, n_max, plan);
    }
    CUtensorMap tq, tk, tv, tkl, tvl;
    if (!encode_q_map(c, &tq, q, R) || !encode_pages_map(c, &tk, k_pages, n_pages) || !encode_pages_map(c, &tv, v_pages, n_pages) ||
        !encode_local_map(c, &tkl, k_local, (long long)n_seqs * k * k) || !encode_local_map(c, &tvl, v_local, (long long)n_seqs * k * k))
      return fail(c, TIDAR_ECUDA, "cuTensorMapEncodeTiled failed for an attention operand");
    const AttnMaps am{&tq, &tk, &tv, &tkl, &tvl, 0, 0};
    if (d.streams) {
      c->route = {d.cluster, d.pieces > 1, 0};
      attn_tc::Args a = attention_args(c, am, g, (bf16 *)out);
      a.direct.seq_len = seq_len; a.direct.k = k; a.direct.n_max = n_max; a.direct.pieces = d.pieces;
      a.direct.per_group = (k * (k + 1) + a.spt - 1) / a.spt;
      const int tiles = n_seqs * a.direct.per_group * a.Hkv;
      if (d.streams == 2) launch_attention_kernel<2, true>(c, tiles * d.pieces, am, a, d.cluster); else launch_attention_kernel<1, true>(c, tiles, am, a);
      if (d.pieces > 1) launch_attention_merge<true>(c, tiles, a);
    } else {
      launch_attention_tc(c, plan, am, g, (bf16 *)out, false, false);   // behind the kernel that makes the plan
    }
  } else {
    {
      Launch l(c, TIDAR_TC_EMBED);
      attn_meta_kernel<<<(R + 127) / 128, 128, 0, c->stream>>>(c->meta, seq_len, k, R, n_max);
    }
    launch_attention(c, (const bf16 *)q, (const bf16 *)k_pages, (const bf16 *)v_pages, g, (const bf16 *)k_local, (const bf16 *)v_local,
                     (bf16 *)out, R);
  }
  CUDA_TRY(c, cudaGetLastError());
  return TIDAR_OK;
}

}  // extern "C"

// =============================================================================
// Attention without any allocation.
//
// Some hosts of this library may not allocate device memory at the moment they
// need attention: a serving process whose memory pool has been handed over
// completely to another component, a real-time loop that must not enter the
// allocator (cudaMalloc can block on every other stream of the device), or a
// plug-in that is given tensors but no allocator.  For them the per-row
// visibility table that tidar_attention keeps in the context arena lives in the
// fixed array below instead.  The array is part of the library image: every GPU
// that loads the library carries it (TIDAR_STATIC_MAX_ROWS * 5 * 4 bytes) until
// the process exits.
// =============================================================================
#define TIDAR_STATIC_MAX_ROWS 4352            /* 16 sequences of 16*17 slots */
#define TIDAR_STATIC_MAX_DEVICES 64

static __device__ __align__(256) int32_t g_static_rowmeta[5 * TIDAR_STATIC_MAX_ROWS];

namespace {
// Device address of g_static_rowmeta per device ordinal.  In host code the symbol's
// name is only a handle; the address a kernel can use comes from cudaGetSymbolAddress
// with that device current.
int32_t *g_static_ptr[TIDAR_STATIC_MAX_DEVICES] = {};
}  // namespace

extern "C" int tidar_attention_static(const void *q, const void *k_pages, const void *v_pages, int32_t n_pages, const int32_t *page_table,
                                      int32_t pages_per_seq, const int32_t *seq_len, const void *k_local, const void *v_local,
                                      void *out, int32_t n_seqs, int32_t k, int32_t n_q_heads, int32_t n_kv_heads,
                                      int32_t head_dim, void *cuda_stream) {
  if (!q || !k_pages || !v_pages || !page_table || !seq_len || !k_local || !v_local || !out)
    return fail(nullptr, TIDAR_EINVAL, "tidar_attention_static: null argument");
  if (head_dim != 64 && head_dim != 128) return fail(nullptr, TIDAR_EINVAL, "tidar_attention_static: head_dim must be 64 or 128");
  if (n_kv_heads < 1 || n_q_heads < 1 || n_q_heads % n_kv_heads)
    return fail(nullptr, TIDAR_EINVAL, "tidar_attention_static: n_q_heads must be a positive multiple of n_kv_heads");
  if (k < 1 || k > 32 || n_seqs < 1 || pages_per_seq < 1 || n_pages < 1)
    return fail(nullptr, TIDAR_EINVAL, "tidar_attention_static: bad k, n_seqs, n_pages or pages_per_seq");
  if ((long long)pages_per_seq * 64 < k) return fail(nullptr, TIDAR_EINVAL, "tidar_attention_static: the page table cannot back the k causal slots");
  // the kernel reads K/V rows with 16-byte loads
  if (((uintptr_t)q | (uintptr_t)k_pages | (uintptr_t)v_pages | (uintptr_t)k_local | (uintptr_t)v_local | (uintptr_t)out) % 16 ||
      ((uintptr_t)page_table | (uintptr_t)seq_len) % 4)
    return fail(nullptr, TIDAR_EINVAL, "tidar_attention_static: tensors must be 16-byte aligned (page_table and seq_len 4-byte)");
  const long long rows = (long long)n_seqs * k * (k + 1);
  if (rows > TIDAR_STATIC_MAX_ROWS)
    return fail(nullptr, TIDAR_ECAPACITY, "tidar_attention_static: %lld rows exceed the built-in table of %d rows; use tidar_attention",
                rows, TIDAR_STATIC_MAX_ROWS);
  int dev = -1;
  CUDA_TRY(nullptr, cudaGetDevice(&dev));
  if (dev < 0 || dev >= TIDAR_STATIC_MAX_DEVICES) return fail(nullptr, TIDAR_EINVAL, "tidar_attention_static: device ordinal %d not supported", dev);
  // First call on this device: resolve the table's device address.  Not synchronised between
  // host threads: two first calls at once both look the address up and store the same value.
  if (!g_static_ptr[dev]) {
    int32_t *p = nullptr;
    CUDA_TRY(nullptr, cudaGetSymbolAddress((void **)&p, g_static_rowmeta));
    if (!p) return fail(nullptr, TIDAR_ECUDA, "tidar_attention_static: no device address for the built-in table");
    g_static_ptr[dev] = p;
  }
  int32_t *base = g_static_ptr[dev];
  const int R = (int)rows;
  RowMeta m{};
  m.seq = base; m.pos = base + TIDAR_STATIC_MAX_ROWS; m.nvis = base + 2 * TIDAR_STATIC_MAX_ROWS;
  m.loc0 = base + 3 * TIDAR_STATIC_MAX_ROWS; m.nloc = base + 4 * TIDAR_STATIC_MAX_ROWS;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  // every entry a row reads is rewritten here for rows [0, R): nothing has to start at zero
  attn_meta_kernel<<<(R + 127) / 128, 128, 0, st>>>(m, seq_len, k, R, pages_per_seq * 64 - k);
  KvGeom g{n_kv_heads, head_dim, 64, pages_per_seq, page_table, n_pages};
  const float scale = 1.0f / sqrtf((float)head_dim);
  dim3 grid(R, n_q_heads);
  if (head_dim == 128)
    attn_replay_kernel<128><<<grid, 32, 0, st>>>((const bf16 *)q, (const bf16 *)k_pages, (const bf16 *)v_pages, g, m, (const bf16 *)k_local,
                                                 (const bf16 *)v_local, (bf16 *)out, n_q_heads, scale);
  else
    attn_replay_kernel<64><<<grid, 32, 0, st>>>((const bf16 *)q, (const bf16 *)k_pages, (const bf16 *)v_pages, g, m, (const bf16 *)k_local,
                                                (const bf16 *)v_local, (bf16 *)out, n_q_heads, scale);
  CUDA_TRY(nullptr, cudaGetLastError());
  return TIDAR_OK;
}
