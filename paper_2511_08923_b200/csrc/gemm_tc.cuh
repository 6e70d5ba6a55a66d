// Small-M weight-streaming GEMM on tcgen05 tensor cores.
//
//   out[r][n] = sum_k A[r][k] * W[n][k]      A [R][K] bf16 (activations, few rows),
//                                            W [N][K] bf16 (weights, streamed once)
//
// A decode step has only k*(k+1) token slots per sequence (paper Section 3.3 footnote),
// so every projection is a GEMM with a small row count and a weight matrix that is read
// exactly once: the regime in which, by the paper's argument, extra token slots are nearly free
// (Section 1; figure "Latency Scaling").  The kernel therefore puts the WEIGHT rows on the TMEM lanes (the MMA M
// dimension) and the activation rows on the MMA N dimension (up to 288 = two instructions
// of up to 144 columns), so no tensor-core work is wasted on padding rows.
//
// PAIR instances: two CTAs (a cluster) share one MMA of M = 256.  Each holds its own 128-row weight tile and HALF of the
// activation rows, and gets the accumulator of its own tile, all columns.  What bounds the main loop of many
// rows is shared memory: for 272 rows a lone CTA reads 66 KB of operands and has 51 KB written to it per 64-wide K
// block, 916 cycles at 128 B per cycle against 544 cycles of MMAs (measured: 811 - 867); half the activations
// leaves 49 + 33 KB, 640 cycles.
// SMALL instances: few rows, see below.
//
// Work item = (row block, weight tile or pair of tiles, K split).  Persistent CTAs, one per SM, loop
// over items.  Warp roles:
//   warp 0      streams the weight tiles by TMA into a ring of stages (a tile comes from HBM and takes > 1 us to arrive);
//   warp 3      streams the activation tiles (from L2) into the same stages;
//   warp 1      issues the MMAs into one fp32 accumulator in TMEM (even CTA of a pair);
//   warp 2      watches the stages' mbarriers on behalf of warp 1, which must not touch the
//               memory pipeline between its MMAs, and releases it through hardware barriers (even CTA);
//   warps 4-11  drain the accumulator into registers (which frees it for the next item at
//               once) and run the epilogue from registers while the next item's MMAs proceed.
#pragma once
#include <algorithm>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace gemm_tc {

constexpr int TILE_N = 128;         // weight rows per tile (TMEM lanes)
constexpr int TILE_K = 64;          // bf16 elements per 128-byte swizzled row
constexpr int MAX_ROWS = 288;       // activation rows of a single row block (2 x 144 TMEM columns)
constexpr int BLOCK_ROWS = 256;     // activation rows of a row block that one instruction covers (see plan_blocks)
constexpr int EPI_WARPS = 8;
constexpr int ROLE_WARPS = 4;      // warpgroup 0: weight producer, MMA issuer, stage watcher, activation producer
constexpr int THREADS = 32 * (ROLE_WARPS + EPI_WARPS);
constexpr int ROLE_REGS = 56, EPI_REGS = 224;   // registers per thread after the split: 128 * 56 + 256 * 224 <= 64 K
constexpr int W_STAGE_BYTES = TILE_N * TILE_K * 2;
constexpr int SMEM_BUDGET = 212 * 1024;   // dynamic shared memory for the ring; up to 9 KB of static shared memory come on top
constexpr int TMEM_COLS = 512;
constexpr int MAX_STAGES = 12;     // of the ring (hardware barriers 1 .. 12)

// Few rows (SMALL instances: a row block of at most SMALL_ROWS).  Such a launch is bound by streaming its weights, but a
// good part of its time used to be spent elsewhere:
// * Before the first weights had arrived: with all of an SM's registers, a CTA could not become resident before the
//   SM had emptied.  A SMALL CTA takes 80 registers per thread and 128 TMEM columns, so it sits beside the kernels
//   between two projections, its ring full of weights by the time its activations are ready.
// * Per stage: each costs its producers, the watcher and the MMA warp some 600 cycles of barrier tests and issue,
//   three times what the MMAs of a 64-wide K block take with few rows.  A stage holds two K blocks there.
// 1.5B-class autoregressive step of 8 rows 1.90 -> 1.75 ms, 8B-class step of 20 rows 4.2 -> 4.0 ms (the gate/up projection
// of the former 11.4 -> 10.3 us, QKV 5.3 -> 3.4 us).  80 registers are not enough for the SwiGLU epilogue, which spills 27 words per thread
// once per item.  Measured and not kept: fetching weights into L2 ahead of the ring, this
// launch's or the next projection's (2 - 8 % slower, the more the further ahead).
constexpr int SMALL_ROWS = 96;
constexpr int SMALL_TMEM_COLS = 128;
__host__ __device__ constexpr int k_per_stage(bool small) { return small ? 2 : 1; }     // K blocks of 64 per stage
__host__ __device__ constexpr int tile_rows(bool small) { return small ? TILE_N : 2 * TILE_N; }   // weight rows of an item

// MODE_SAMPLE is MODE_ARGMAX with Gumbel noise added to the tempered logits (a draw per row instead of
// the argmax); it is a mode of its own so that the greedy LM head carries none of its registers.
// MODE_LSE (likelihood scoring): the logits never leave the chip; each warp of each tile leaves, per row, the maximum of its 32 logits and
// the sum of their exponentials below it, and the lane that owns a row's target id leaves that logit.  No state is carried from
// tile to tile, so the row block varies fastest as in the projections and a weight tile is read once from HBM.
enum Mode { MODE_SLAB = 0, MODE_SWIGLU = 1, MODE_ARGMAX = 2, MODE_SAMPLE = 3, MODE_LSE = 4 };

// A "tile" below is what an item covers: tile_rows(small) weight rows.
struct Args {
  int R, N, K;              // activation rows in use, output features, input features
  int rb_rows;              // rows per row block: multiple of 16, 16..288
  int n_rb;                 // row blocks
  int n_tiles;              // ceil(N / tile rows)
  int S;                    // K splits of the split region
  int fused_items;          // items [0, fused_items) are whole tiles 0.. (no K split) finished by the mode's own epilogue;
                            // the rest are tiles tile_b0.. split S ways along K, written as fp32 slabs
  int tile_b0, n_tiles_b;   // first tile and tile count of the split region
  int kb_total;             // stages of K: K / 64, or half of it (rounded up) in a SMALL launch
  int stages;               // depth of the ring (<= MAX_STAGES)
  int n1, n2;               // MMA N of the two instructions (n2 may be 0)
  // MODE_SLAB: out[split][r][n], fp32 or (slab_bf16) bf16; strides in elements
  // accumulate (S = 1 only): out is added to instead of written; every element has one writer, so the result does not
  // depend on any order
  void *out; long long slab_stride; int ldo; int slab_bf16, accumulate;
  // MODE_SWIGLU: weight rows interleave (gate f, up f); H[r][f] = silu(gate) * up, bf16
  bf16 *H; int ldh;
  // MODE_ARGMAX: per (CTA, lane quadrant) candidates, [R][cand_ld >= gridDim*4] (index -1 = none; the
  // caller pre-fills the index table with -1); optional fp32 dump [R][ld_dump]
  float *cand_val; int32_t *cand_idx; int cand_ld; float *dump; int ld_dump; int col0;
  // MODE_SAMPLE: the compared value is logit * inv_temp + Gumbel noise of (skey[row], id),
  // i.e. a draw from softmax(logits / temperature) per row (see gumbel_noise); the dump keeps the raw logits
  float inv_temp; const uint32_t *skey;
  // MODE_LSE: (max, sum) of lse_parts(N) groups of 32 ids, [group][R]; the target id of each row, and its logit
  float2 *lse; const int32_t *target; float *tgt_logit;
  int warm_epilogue;        // walk through the epilogue once before the first accumulator is ready (see the kernel)
  int *status;              // device word set to 1 when a bounded wait gave up
  __host__ __device__ int tile_b0_or_all() const { return n_tiles_b ? tile_b0 : n_tiles; }   // tiles per row block in the fused region
  __host__ __device__ int total_items() const { return fused_items + n_rb * n_tiles_b * S; }
};

__host__ __device__ inline int lse_parts(int N) { return (N + tile_rows(false) - 1) / tile_rows(false) * (tile_rows(false) / 32); }

struct Item { int rb, tile, split, kb0, kb1; bool fused; };
// Item order.  With several row blocks (a long first pass) the row block varies fastest: the CTAs
// that run side by side then work on the SAME weight tile for different rows, so the tile comes
// from HBM once and from L2 for the others, and the pass is bound by the tensor cores instead of
// streaming every weight matrix once per row block.  The LM-head mode keeps a row block's tiles
// together instead (tile fastest): its epilogue carries a running argmax per row block.
template <int MODE>
__device__ __forceinline__ Item decode_item(const Args &g, int item) {
  Item w;
  if (item < g.fused_items) {
    w.fused = true; w.split = 0;
    if (MODE == MODE_ARGMAX || MODE == MODE_SAMPLE) { w.tile = item % g.tile_b0_or_all(); w.rb = item / g.tile_b0_or_all(); }
    else { w.rb = item % g.n_rb; w.tile = item / g.n_rb; }
    w.kb0 = 0; w.kb1 = g.kb_total;
  } else {
    const int j = item - g.fused_items;
    w.fused = false; w.rb = j % g.n_rb; w.split = (j / g.n_rb) % g.S; w.tile = g.tile_b0 + j / (g.n_rb * g.S);
    w.kb0 = (int)((long long)g.kb_total * w.split / g.S); w.kb1 = (int)((long long)g.kb_total * (w.split + 1) / g.S);
  }
  return w;
}

// silu(g) * u.  The fast division is exact enough for a bf16 result (2 ulp of fp32) and returns
// the right limit (-0) when exp(-g) overflows.
__device__ __forceinline__ float silu_mul(float g, float u) { return __fdividef(g, 1.f + __expf(-g)) * u; }

// PAIR: two CTAs share an item (see the head of this file); otherwise SMALL.
template <int MODE, bool SMALL = false>
__global__ void __launch_bounds__(THREADS, SMALL ? 2 : 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmA, const Args g, const TlSlot tl) {
  constexpr bool PAIR = !SMALL;
  constexpr int KPS = k_per_stage(SMALL);
  constexpr int NCH = SMALL ? SMALL_ROWS / 32 : 9;         // 16-column chunks of the accumulator per epilogue warp
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[MAX_STAGES], empty[MAX_STAGES], tmem_full_bar, tmem_empty_bar;
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;
  __shared__ __align__(16) uint16_t epi_stage[MODE == MODE_SWIGLU ? EPI_WARPS : 1][32][16];   // MODE_SWIGLU: two 16-column chunks per epilogue warp, [column][feature]

  const int warp = sm100::warp_index(), lane = threadIdx.x & 31;
  const int rank = PAIR ? (int)sm100::cluster_rank() : 0;
  const int worker = PAIR ? blockIdx.x >> 1 : blockIdx.x, n_workers = PAIR ? gridDim.x >> 1 : gridDim.x;
  const uint32_t smem0 = (sm100::smem_u32(smem_raw) + 1023u) & ~1023u;
  // A stage: KPS weight blocks [128][64], then KPS activation blocks [a_rows][64] (a_rows multiple of 8: whole swizzle atoms).
  const int a_rows = PAIR ? g.rb_rows >> 1 : g.rb_rows;
  const uint32_t a_block = (uint32_t)(a_rows * TILE_K * 2);
  const uint32_t stage_bytes = KPS * (W_STAGE_BYTES + a_block);
  const int n_items = g.total_items();

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < MAX_STAGES; ++s) { sm100::mbar_init(sm100::smem_u32(&full[s]), 1); sm100::mbar_init(sm100::smem_u32(&empty[s]), 1); }
    sm100::mbar_init(sm100::smem_u32(&tmem_full_bar), 1);
    sm100::mbar_init(sm100::smem_u32(&tmem_empty_bar), PAIR ? 2 * EPI_WARPS : EPI_WARPS);
    sm100::fence_mbar_init();
  }
  if (warp == 1) {
    __syncwarp();
    if constexpr (PAIR) { sm100::tmem_alloc_pair(sm100::smem_u32(&tmem_base_slot), TMEM_COLS); sm100::tmem_relinquish_pair(); }
    else { sm100::tmem_alloc(sm100::smem_u32(&tmem_base_slot), SMALL_TMEM_COLS); sm100::tmem_relinquish(); }
  }
  sm100::tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) sm100::cluster_sync();     // the other CTA's barriers exist
  sm100::tc_fence_after();
  const uint32_t tmem_acc = tmem_base_slot;
  // Only now may the next kernel's CTAs be scheduled: one that got in before this CTA had its tensor memory could take
  // it, and would keep it while it waits for this kernel.
  pdl_trigger();
  volatile int *abortp = &abort_flag;

  // The epilogue warps hold the whole accumulator (144 registers per thread) next to their
  // own arithmetic; at the kernel-wide limit of 168 the compiler serialises that arithmetic to
  // save registers (SwiGLU: 1000 instead of 300 cycles per chunk) and spills in the argmax.  The
  // four role warps need few registers, so their warpgroup hands most of its share over.
  // (Each reallocation heads the code that runs under it, which is how the compiler learns
  // the register budget of that code.)

  if (warp < ROLE_WARPS) {
  if constexpr (!SMALL) sm100::setmaxnreg_dec<ROLE_REGS>();
  if (warp == 0 || warp == 3) {
    // ===================== weight producer (warp 0), activation producer (warp 3) =====================
    // Both fill the same stages.  A stage's bytes (of both CTAs of a pair) are counted on the even CTA's barrier, where the weight
    // producer announces them; loads that complete before the announcement are no problem, the phase needs its arrival too.
    // Weights are never written by a kernel, so their producer does not wait for the previous kernel:
    // the ring fills while that kernel is still finishing.
    // (The whole warp walks the schedule and one elected lane issues: see the MMA issuer.)
    const bool is_w = warp == 0;
    const CUtensorMap *tm = is_w ? &tmW : &tmA;
    if (lane == 0) sm100::prefetch_tensormap(tm);
    const uint64_t pol = is_w ? sm100::policy_evict_first() : sm100::policy_evict_last();
    int s = 0; uint32_t ph = 0; bool ok = true;
    if (!is_w) {
      pdl_wait();                      // the activations are the previous kernel's output
      if (lane == 0) tl_go(tl);
    }
    for (int item = worker; item < n_items && ok; item += n_workers) {
      const Item w = decode_item<MODE>(g, item);
      const int row = is_w ? (PAIR ? (w.tile * 2 + rank) * TILE_N : w.tile * TILE_N) : w.rb * g.rb_rows + rank * a_rows;
      for (int kb = w.kb0; kb < w.kb1; ++kb) {
        if (!sm100::mbar_wait_warp(sm100::smem_u32(&empty[s]), ph ^ 1u, abortp)) { ok = false; break; }
        if (sm100::elect_one()) {
          const uint32_t fb = sm100::smem_u32(&full[s]);
          const uint32_t dst = smem0 + (uint32_t)s * stage_bytes + (is_w ? 0u : (uint32_t)(KPS * W_STAGE_BYTES));
          if (is_w && rank == 0) sm100::mbar_expect_tx(fb, (PAIR ? 2u : 1u) * stage_bytes);
          if constexpr (PAIR) sm100::tma_load_2d_pair(dst, tm, sm100::cluster_addr(fb, 0), kb * TILE_K, row, pol);
          else sm100::tma_load_3d(dst, tm, fb, 0, row, kb * KPS, pol);
        }
        __syncwarp();
        if (++s == g.stages) { s = 0; ph ^= 1u; }
      }
    }
  } else if (warp == 1 && rank == 0) {
    // ===================== MMA issuer =====================
    // One thread issues every MMA.  The whole warp runs the loop, with a warp index that the compiler can see is uniform, and elects the
    // thread: with the operands in uniform registers an MMA issues in 59 cycles, behind a plain test of the lane
    // index in 90 (a K block of 272 rows: 715 instead of 543 cycles).  That is barely faster than the tensor pipe
    // retires them, so nothing else may sit in this instruction stream: a test of an mbarrier
    // (any access through the memory pipeline) completes only once the MMAs queued before it
    // have gone out, and the pipe runs dry for ~250 cycles per K block.  The watcher warp
    // therefore does the mbarrier waits and releases this warp through one hardware barrier
    // per stage.  Descriptors are built once and advanced with plain adds (the start-address
    // field counts 16-byte units and never carries out of its 14 bits inside shared memory).
    //
    // This warp and the watcher run the same (item, K block) schedule to the end whatever
    // happens elsewhere, one barrier operation each per K block, so neither can be left
    // waiting for the other; after a failed wait the MMAs read stale tiles, which is harmless,
    // and the status word reports the failure.
    constexpr int M = PAIR ? 2 * TILE_N : TILE_N;
    const uint32_t idesc1 = sm100::make_idesc_bf16(M, g.n1), idesc2 = sm100::make_idesc_bf16(M, g.n2 ? g.n2 : 16);
    const uint64_t wdesc0 = sm100::make_desc_sw128(smem0), adesc0 = sm100::make_desc_sw128(smem0 + KPS * W_STAGE_BYTES);   // stage 0
    const uint64_t stage16 = (uint64_t)(stage_bytes >> 4), a_block16 = (uint64_t)(a_block >> 4);
    const uint64_t a2_off16 = (uint64_t)((PAIR ? g.n1 >> 1 : g.n1) * 8);
    const uint32_t tmem_acc2 = tmem_acc + (uint32_t)g.n1;
    const bool two = g.n2 != 0;
    auto mma = [](uint32_t d, uint64_t wd, uint64_t ad, uint32_t idesc, uint32_t acc) {
      if constexpr (PAIR) sm100::mma_bf16_ss_pair(d, wd, ad, idesc, acc); else sm100::mma_bf16_ss(d, wd, ad, idesc, acc);
    };
    auto commit = [](uint32_t bar) { if constexpr (PAIR) sm100::mma_commit_pair(bar); else sm100::mma_commit(bar); };
    int s = 0;
    uint64_t wd = wdesc0, ad = adesc0;
    for (int item = worker; item < n_items; item += n_workers) {
      const Item w = decode_item<MODE>(g, item);
      uint32_t acc = 0u;                 // the watcher's first release of an item also says that the accumulator is free
      for (int kb = w.kb0; kb < w.kb1; ++kb) {
        sm100::named_bar_sync(1u + (uint32_t)s, 64);
        sm100::tc_fence_after();
        if (sm100::elect_one()) {
          if (PAIR && two) {
            const uint64_t ad2 = ad + a2_off16;
#pragma unroll
            for (int kk = 0; kk < TILE_K / 16; ++kk) {
              mma(tmem_acc, wd + 2 * kk, ad + 2 * kk, idesc1, acc);
              mma(tmem_acc2, wd + 2 * kk, ad2 + 2 * kk, idesc2, acc);
              acc = 1u;
            }
          } else {
#pragma unroll
            for (int kk = 0; kk < KPS * TILE_K / 16; ++kk) {
              mma(tmem_acc, wd + (kk / 4) * (W_STAGE_BYTES >> 4) + 2 * (kk % 4), ad + (kk / 4) * a_block16 + 2 * (kk % 4), idesc1, acc);
              acc = 1u;
            }
          }
          commit(sm100::smem_u32(&empty[s]));       // the stage is reusable once these MMAs have read it
        }
        __syncwarp();
        acc = 1u;
        wd += stage16; ad += stage16;
        if (++s == g.stages) { s = 0; wd = wdesc0; ad = adesc0; }
      }
      if (sm100::elect_one()) commit(sm100::smem_u32(&tmem_full_bar));
      __syncwarp();
    }
  } else if (warp == 2 && rank == 0) {
    // ===================== stage watcher =====================
    // Waits (bounded) for the accumulator to be drained and for each stage's loads to land,
    // then arrives on the stage's hardware barrier.  A stage's barrier cannot be arrived on
    // twice before the MMA warp has passed it: the second landing needs the producer's refill,
    // which needs the MMA warp's commit for the first.  After a failed wait that argument no
    // longer holds, so from then on the watcher meets the MMA warp at every barrier instead.
    int s = 0; uint32_t ph = 0, it = 0; bool failed = false;
    for (int item = worker; item < n_items; item += n_workers, ++it) {
      const Item w = decode_item<MODE>(g, item);
      if (!failed) {
        bool ok = true;
        if (lane == 0) ok = sm100::mbar_wait(sm100::smem_u32(&tmem_empty_bar), (it & 1u) ^ 1u, abortp);
        failed = !__shfl_sync(0xffffffffu, ok, 0);
      }
      for (int kb = w.kb0; kb < w.kb1; ++kb) {
        if (!failed) {
          bool ok = true;
          if (lane == 0) ok = sm100::mbar_wait(sm100::smem_u32(&full[s]), ph, abortp);
          failed = !__shfl_sync(0xffffffffu, ok, 0);
        }
        if (!failed) sm100::named_bar_arrive(1u + (uint32_t)s, 64);
        else sm100::named_bar_sync(1u + (uint32_t)s, 64);
        if (++s == g.stages) { s = 0; ph ^= 1u; }
      }
    }
  }
  } else {
    if constexpr (!SMALL) sm100::setmaxnreg_inc<EPI_REGS>();
    // ===================== epilogue =====================
    pdl_wait();
    const int q = warp & 3;                      // TMEM lane quadrant this warp may read
    const int half = (warp - ROLE_WARPS) >> 2;
    const int hc = ((g.rb_rows / 2 + 15) / 16) * 16;
    const int c_begin = half ? hc : 0;
    const int c_end = half ? g.rb_rows : (hc < g.rb_rows ? hc : g.rb_rows);
    const int ncols = c_end - c_begin;           // multiple of 16, <= 144
    // Row of the block that accumulator column c (a multiple of 8, or any column of its group of 8) belongs to.  With two instructions over
    // a pair, the first takes the first n1 / 2 of each CTA's rows and the second the rest.
    const int h1 = g.n1 >> 1, h2 = g.n2 >> 1;
    auto col_row = [&](int c) {
      if (!PAIR || h2 == 0) return c;
      return c < h1 ? c : c < 2 * h1 ? c + h2 : c < 2 * h1 + h2 ? c - h1 : c;
    };
    const uint32_t drained_bar = PAIR ? sm100::cluster_addr(sm100::smem_u32(&tmem_empty_bar), 0) : sm100::smem_u32(&tmem_empty_bar);
    auto drained = [&]() {                       // the accumulator may be overwritten
      sm100::tc_fence_before();
      __syncwarp();
      if (lane == 0) { if constexpr (PAIR) sm100::mbar_arrive_cluster(drained_bar); else sm100::mbar_arrive(drained_bar); }
    };
    uint32_t it = 0; bool ok = true;
    // Wait for the accumulator; the lanes leave together, but each with an answer of its own.  After a wait that gave up the item is gone through all the
    // same, on stale values (all of a warp's lanes take part in its tensor-memory accesses, and the status word reports the failure): the
    // lanes agree behind the item (`next`), for a vote here would stand in the way of every item (1.5B-class step: 0.1 % longer).
    auto wait_full = [&](uint32_t n) { return sm100::mbar_wait_converged(sm100::smem_u32(&tmem_full_bar), n & 1u, abortp); };
    auto next = [&](int item) { ok = __all_sync(0xffffffffu, ok) != 0; ++it; return item + n_workers; };
    // MODE_ARGMAX: running best of column c_begin + 32*slot + lane, and the row block it belongs to
    float best_v[5]; int best_i[5]; int cur_rb = -1;
#pragma unroll
    for (int k = 0; k < 5; ++k) { best_v[k] = -INFINITY; best_i[k] = 0x7fffffff; }
    auto flush_best = [&]() {
      if (cur_rb < 0) return;
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const int cidx = k * 32 + lane;
        const int r = cur_rb * g.rb_rows + col_row(c_begin + cidx);
        if (cidx < ncols && r < g.R) {
          const long long o = (long long)r * g.cand_ld + (blockIdx.x * 4 + q);
          g.cand_val[o] = best_v[k]; g.cand_idx[o] = best_i[k] == 0x7fffffff ? -1 : best_i[k];
        }
        best_v[k] = -INFINITY; best_i[k] = 0x7fffffff;
      }
    };
    // ---- MODE_SWIGLU: two 16-column chunks of the accumulator -> bf16 rows of H ----
    // Lane pairs (2j, 2j+1) hold gate and up of feature n/2; the even lane finishes
    // column c, the odd lane column c+1, after one exchange per column pair.  The
    // results of a 16-column chunk (16 columns x 16 features per warp) are turned
    // through shared memory so that every lane stores 8 consecutive features of one
    // row with one 16-byte store: 2-byte stores from each lane took 18 us per tile.
    // All exchanges first, then sixteen independent silu chains (one chain at a time is bound by
    // instruction latency: 16 us per tile instead of 2), then the turn through shared memory.
    // c0 / c1: the two chunks (c1 only if second); col0: accumulator column of c0's first; row_block: first row of the block;
    // n0: first weight row of the tile.
    auto swiglu_pass = [&](const uint32_t (&c0)[16], const uint32_t (&c1)[16], bool second, int col0, int row_block, int R_live, int n0) {
      const bool odd = lane & 1;
      uint16_t (*stage)[16] = epi_stage[MODE == MODE_SWIGLU ? warp - ROLE_WARPS : 0];
      const int srow = lane >> 1, sf = (lane & 1) * 8;
      const int f0 = ((n0 + q * 32) >> 1) + sf;          // first of this lane's 8 features
      const int n_feat = g.N >> 1;
      float h[2][8];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (c == 0 || second) {
          uint32_t recv[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) recv[j] = __shfl_xor_sync(0xffffffffu, odd ? (c ? c1[2 * j] : c0[2 * j]) : (c ? c1[2 * j + 1] : c0[2 * j + 1]), 1);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float gate = __uint_as_float(odd ? recv[j] : (c ? c1[2 * j] : c0[2 * j]));
            const float up = __uint_as_float(odd ? (c ? c1[2 * j + 1] : c0[2 * j + 1]) : recv[j]);
            h[c][j] = silu_mul(gate, up);
          }
        }
      }
#pragma unroll
      for (int c = 0; c < 2; ++c)
        if (c == 0 || second) {
#pragma unroll
          for (int j = 0; j < 8; ++j) stage[c * 16 + 2 * j + (odd ? 1 : 0)][lane >> 1] = __bfloat16_as_ushort(__float2bfloat16(h[c][j]));
        }
      __syncwarp();
#pragma unroll
      for (int c = 0; c < 2; ++c)
        if (c == 0 || second) {
          const uint4 packed = *reinterpret_cast<const uint4 *>(&stage[c * 16 + srow][sf]);
          const int r = row_block + col_row(col0 + c * 16 + srow);
          if (r < R_live) {
            bf16 *dst = g.H + (long long)r * g.ldh + f0;
            if (f0 + 8 <= n_feat && (g.ldh & 7) == 0) {
              *reinterpret_cast<uint4 *>(dst) = packed;
            } else {
              const uint16_t *e = reinterpret_cast<const uint16_t *>(&packed);
              for (int t = 0; t < 8; ++t)
                if (f0 + t < n_feat) dst[t] = __ushort_as_bfloat16(e[t]);
            }
          }
        }
      __syncwarp();
    };
    // The epilogue below is long straight-line code that a CTA runs once or twice, and between two
    // launches of this kernel the other kernels of a layer push it out of the instruction cache: run
    // cold, next to the MMAs of the next item, one SwiGLU pass took 2 - 3.5 us instead of 0.4.  These
    // warps have nothing to do while the first item's MMAs run, so they first walk through the
    // epilogue once with every store and barrier operation switched off (dry), which
    // brings the code in; g.warm_epilogue is a run-time value so that both walks share one copy.
    // Slabs and additions to the residual stream of the pair instances are walked through as well, where every worker has one item that is long enough (see plan_gemm): 272 rows x 128 features leave a CTA in 3.6 - 3.9 us
    // then (4.6 - 6.4 before; 3.4 in a kernel that does nothing else, 28 B per cycle: the SM's port, whatever the instruction).  That walk
    // starts a little later, for the role warps' first rounds fetch code too (started at once, the first stage landed 0.3 us later).  Turning them
    // into a short loop over tensor memory instead was slower (8.3 us): a store holds its register until the port takes it.
    // The SMALL instances' slabs are too short for a walk (it cost as much as it gave).
    // A fused item that is its CTA's last one takes a third route: nobody waits for the accumulator, so it
    // stays in tensor memory and a loop of a few hundred instructions takes 32 columns per round (the
    // 1.5B-class gate/up projection, one item per CTA, ends 4 us earlier than with the long code).  With few rows
    // every fused item goes that way: it is one or two rounds.  So does a split item of a SwiGLU launch, 16 columns per round.  Their first round
    // is a dry one, on whatever tensor memory holds, before the wait for the accumulator (8B-class gate/up at 20 rows 33.3 -> 30.3 us, at 272 rows
    // 47.9 -> 46).
    const bool may_walk = !SMALL && g.warm_epilogue != 0;
    bool walk = may_walk && (MODE == MODE_SLAB || (MODE == MODE_SWIGLU && worker + n_workers < n_items));
    for (int item = worker; item < n_items && ok;) {
      const Item w = decode_item<MODE>(g, item);
      const int split = w.split, rb = w.rb, row_block = rb * g.rb_rows;
      const int n0 = (PAIR ? w.tile * 2 + rank : w.tile) * TILE_N;      // first weight row of this CTA's tile
      if (MODE == MODE_SWIGLU && w.fused && (SMALL || item + n_workers >= n_items)) {
        const uint32_t t0 = tmem_acc + ((uint32_t)(q * 32) << 16) + (uint32_t)c_begin;
        bool live = false;
#pragma unroll 1
        for (int cc = 0; !live || cc < ncols;) {       // (a warp without columns waits for the accumulator too, or it would run ahead of the others)
          uint32_t c0[16], c1[16];
          const bool second = cc + 16 < ncols;
          sm100::tmem_ld16(t0 + cc, c0);
          if (second) sm100::tmem_ld16(t0 + cc + 16, c1);
          sm100::tmem_wait_ld();
          swiglu_pass(c0, c1, second, c_begin + cc, row_block, live ? g.R : 0, n0);
          if (live) { cc += 32; continue; }
          ok = wait_full(it);
          sm100::tc_fence_after();
          live = true;
        }
        drained();
        item = next(item);
        continue;
      }
      if (MODE == MODE_SWIGLU && !w.fused && !g.slab_bf16) {
        // Partial sums of a split tile (always its CTA's last item).
        const int n = n0 + q * 32 + lane, n_rows = n < g.N ? g.R : 0;
        float *out = reinterpret_cast<float *>(g.out) + (long long)split * g.slab_stride + (n - g.tile_b0 * tile_rows(SMALL));
        const uint32_t t0 = tmem_acc + ((uint32_t)(q * 32) << 16) + (uint32_t)c_begin;
        bool live = false;
#pragma unroll 1
        for (int cc = 0; !live || cc < ncols;) {
          uint32_t c0[16];
          sm100::tmem_ld16(t0 + cc, c0);
          sm100::tmem_wait_ld();
#pragma unroll
          for (int h = 0; h < 16; h += 8) {
            const int r0 = row_block + col_row(c_begin + cc + h);
            float *p = out + (long long)r0 * g.ldo;
            const int rows_left = live ? n_rows - r0 : 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) { if (j < rows_left) *p = __uint_as_float(c0[h + j]); p += g.ldo; }
          }
          if (live) { cc += 16; continue; }
          ok = wait_full(it);
          sm100::tc_fence_after();
          live = true;
        }
        drained();
        item = next(item);
        continue;
      }
      const bool dry = walk;
      if (MODE == MODE_SLAB && dry) __nanosleep(1500);
      uint32_t v[NCH][16];
      if (!dry) {
        ok = wait_full(it);
        sm100::tc_fence_after();
        const uint32_t t0 = tmem_acc + ((uint32_t)(q * 32) << 16) + (uint32_t)c_begin;
#pragma unroll
        for (int i = 0; i < NCH; ++i)
          if (i * 16 < ncols) sm100::tmem_ld16(t0 + i * 16, v[i]);
        sm100::tmem_wait_ld();
        drained();                                       // accumulator free for the next item
      }                                                  // (dry: v holds whatever the registers held; nothing of it is stored)
      const int R_live = dry ? 0 : g.R;                  // rows this walk may store

      const int n = n0 + q * 32 + lane;                  // this thread's output feature
      if (MODE == MODE_SLAB || !w.fused) {
        // split-K partial sums; columns are counted from the first tile of the split region
        const int nc = n - g.tile_b0 * tile_rows(SMALL);
        const bool n_ok = n < g.N;
        if (MODE == MODE_SLAB && g.accumulate) {
          constexpr int RUN = SMALL ? 16 : 8;            // columns that are consecutive rows
          float *out = reinterpret_cast<float *>(g.out) + nc;
#pragma unroll
          for (int i = 0; i < NCH; ++i) {
            if (i * 16 < ncols) {
#pragma unroll
              for (int h = 0; h < 16; h += RUN) {
                const int r0 = row_block + col_row(c_begin + i * 16 + h);
                float *p = out + (long long)r0 * g.ldo;
                const int rows_left = n_ok ? R_live - r0 : 0;
#pragma unroll
                for (int j = 0; j < RUN; ++j) {
                  if (j < rows_left) atomicAdd(p, __uint_as_float(v[i][h + j]));
                  p += g.ldo;
                }
              }
            }
          }
        } else if (MODE == MODE_SLAB && !g.slab_bf16) {
          // One running pointer and a bound counted from the first row of eight: with the address
          // and the row test recomputed per store (r * ldo, r < R) the same 144 stores take 1.65 times
          // as long (19.5 instead of 32 bytes per cycle and SM, the rate the L2 takes stores at).
          float *out = reinterpret_cast<float *>(g.out) + (long long)split * g.slab_stride + nc;
#pragma unroll
          for (int i = 0; i < NCH; ++i) {
            if (i * 16 < ncols) {
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const int r0 = row_block + col_row(c_begin + i * 16 + h * 8);
                float *p = out + (long long)r0 * g.ldo;
                const int rows_left = n_ok ? R_live - r0 : 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  if (j < rows_left) *p = __uint_as_float(v[i][h * 8 + j]);
                  p += g.ldo;
                }
              }
            }
          }
        } else {
          // bf16: lane pairs (2j, 2j+1) exchange so that the even lane stores features
          // (n, n+1) of column c and the odd lane those of column c+1, 4 bytes each
          bf16 *o = reinterpret_cast<bf16 *>(g.out) + (long long)split * g.slab_stride + (nc & ~1);
          const bool odd = lane & 1;
#pragma unroll
          for (int i = 0; i < NCH; ++i) {
            if (i * 16 < ncols) {
#pragma unroll
              for (int j = 0; j < 16; j += 2) {
                const uint32_t send = odd ? v[i][j] : v[i][j + 1];
                const uint32_t recv = __shfl_xor_sync(0xffffffffu, send, 1);
                const float lo = __uint_as_float(odd ? recv : v[i][j]);          // feature n & ~1
                const float hi = __uint_as_float(odd ? v[i][j + 1] : recv);      // feature n | 1
                const int r = row_block + col_row(c_begin + i * 16 + j) + (odd ? 1 : 0);
                if (n_ok && r < R_live) {
                  __nv_bfloat162 h2 = __floats2bfloat162_rn(lo, hi);
                  *reinterpret_cast<__nv_bfloat162 *>(o + (long long)r * g.ldo) = h2;
                }
              }
            }
          }
        }
      } else if (MODE == MODE_SWIGLU && !SMALL) {
        // Register-staged walk over the whole accumulator, two 16-column chunks per pass.
#pragma unroll
        for (int ip = 0; ip < (NCH + 1) / 2; ++ip) {
          if (ip * 32 < ncols) {
            const bool second = (2 * ip + 1) < NCH && (2 * ip + 1) * 16 < ncols;    // warp-uniform
            swiglu_pass(v[2 * ip], v[(2 * ip + 1) < NCH ? 2 * ip + 1 : NCH - 1], second, c_begin + ip * 32, row_block, R_live, n0);
          }
        }
      } else if (MODE == MODE_ARGMAX || MODE == MODE_SAMPLE) {
        // Per column: best (value, index) over the 32 features of this warp, folded into a
        // running best over all tiles this CTA processes.  The 32 lanes x 32 columns of a
        // group are reduced by recursive halving: in the step with stride h a lane keeps the
        // columns whose bit h equals its own lane bit h and hands the others to lane ^ h, so
        // after five steps lane l holds the result of column 32*g + l (31 exchanges per 32
        // columns instead of 160).  Lowest index wins ties, NaN never wins.
        if (rb != cur_rb) { flush_best(); cur_rb = rb; }
        const bool n_ok = n < g.N;
        const int my_idx = (n_ok ? g.col0 + n : 0x7fffffff);
        if (g.dump && n_ok) {
#pragma unroll
          for (int i = 0; i < NCH; ++i)
            if (i * 16 < ncols) {
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const int r = row_block + col_row(c_begin + i * 16 + j);
                if (r < g.R) g.dump[(long long)r * g.ld_dump + n] = __uint_as_float(v[i][j]);
              }
            }
        }
#pragma unroll
        for (int grp = 0; grp < (NCH + 1) / 2; ++grp) {
          if (grp * 32 < ncols) {
            float val[32]; int idx[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              const int i = grp * 2 + (j >> 4);
              float x = (i < NCH && i * 16 < ncols) ? __uint_as_float(v[i < NCH ? i : NCH - 1][j & 15]) : -INFINITY;
              if (MODE == MODE_SAMPLE) {
                const int r = row_block + col_row(c_begin + grp * 32 + j);
                if (r < g.R && n_ok) x = x * g.inv_temp + gumbel_noise(g.skey[r], (uint32_t)my_idx);
              }
              const bool ok_v = n_ok && (x == x);
              val[j] = ok_v ? x : -INFINITY; idx[j] = ok_v ? my_idx : 0x7fffffff;
            }
#pragma unroll
            for (int h = 16; h >= 1; h >>= 1) {
              const bool up = lane & h;
#pragma unroll
              for (int j = 0; j < h; ++j) {
                // columns j (bit h clear) and j + h (bit h set) of the current, already folded, set
                const float sv = up ? val[j] : val[j + h];
                const int si = up ? idx[j] : idx[j + h];
                const float ov = __shfl_xor_sync(0xffffffffu, sv, h);
                const int oi = __shfl_xor_sync(0xffffffffu, si, h);
                const float mv = up ? val[j + h] : val[j];
                const int mi = up ? idx[j + h] : idx[j];
                const bool take = ov > mv || (ov == mv && oi < mi);
                val[j] = take ? ov : mv; idx[j] = take ? oi : mi;
              }
            }
            if (val[0] > best_v[grp] || (val[0] == best_v[grp] && idx[0] < best_i[grp])) { best_v[grp] = val[0]; best_i[grp] = idx[0]; }
          }
        }
      }
      else if (MODE == MODE_LSE) {
        const bool n_ok = n < g.N;
        float2 *out = g.lse + (long long)((n0 + q * 32) >> 5) * g.R;
#pragma unroll
        for (int grp = 0; grp < (NCH + 1) / 2; ++grp) {
          if (grp * 32 < ncols) {
            // lane l finishes column 32 * grp + l
            const int r = row_block + col_row(c_begin + grp * 32 + lane);
            const bool live = grp * 32 + lane < ncols && r < g.R;
            float val[32], mx[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              const int i = grp * 2 + (j >> 4);
              val[j] = n_ok && i < NCH && i * 16 < ncols ? __uint_as_float(v[i < NCH ? i : NCH - 1][j & 15]) : -INFINITY;
              mx[j] = val[j];
            }
            const int tg = live ? g.target[r] - (n0 + q * 32) : -1;
            for (uint32_t hit = __ballot_sync(0xffffffffu, tg >= 0 && tg < 32); hit; hit &= hit - 1) {      // (rare)
              const int j = __ffs(hit) - 1, owner = __shfl_sync(0xffffffffu, tg, j), row = __shfl_sync(0xffffffffu, r, j);
              float x = 0.f;
#pragma unroll
              for (int jj = 0; jj < 32; ++jj) if (jj == j) x = val[jj];
              if (lane == owner) g.tgt_logit[row] = x;
            }
            // maximum and sum over the lanes by recursive halving, as in MODE_ARGMAX
#pragma unroll
            for (int h = 16; h >= 1; h >>= 1) {
              const bool up = lane & h;
#pragma unroll
              for (int j = 0; j < h; ++j) mx[j] = fmaxf(up ? mx[j + h] : mx[j], __shfl_xor_sync(0xffffffffu, up ? mx[j] : mx[j + h], h));
            }
            const float ref = mx[0] == -INFINITY ? 0.f : mx[0];
#pragma unroll
            for (int j = 0; j < 32; ++j) val[j] = __expf(val[j] - __shfl_sync(0xffffffffu, ref, j));
#pragma unroll
            for (int h = 16; h >= 1; h >>= 1) {
              const bool up = lane & h;
#pragma unroll
              for (int j = 0; j < h; ++j) val[j] = (up ? val[j + h] : val[j]) + __shfl_xor_sync(0xffffffffu, up ? val[j] : val[j + h], h);
            }
            if (live) out[r] = make_float2(mx[0], val[0]);
          }
        }
      }
      if (walk) walk = false;                            // the same item again, for real
      else item = next(item);
    }
    if (MODE == MODE_ARGMAX || MODE == MODE_SAMPLE) flush_best();
  }

  // ---- teardown ----
  sm100::tc_fence_before();
  __syncthreads();
  if (abort_flag) {
    if (threadIdx.x == 0 && g.status) atomicExch(g.status, 1);
    // give copies and MMAs that are still in flight time to land before the CTA's
    // shared and tensor memory are released
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    __syncthreads();
  }
  if constexpr (PAIR) sm100::cluster_sync();     // nothing of the other CTA refers to this one any more
  if (warp == 1) {
    __syncwarp();
    sm100::tc_fence_after();
    if constexpr (PAIR) sm100::tmem_dealloc_pair(tmem_acc, TMEM_COLS); else sm100::tmem_dealloc(tmem_acc, SMALL_TMEM_COLS);
  }
  if (threadIdx.x == 0) tl_end(tl);
}

// ---- host side ----------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// bf16 row-major [rows][cols] matrix, box = box_rows x 64 columns, 128-byte swizzle,
// out-of-range elements read as zero.
inline CUresult encode_2d(EncodeTiledFn fn, CUtensorMap *tm, const void *base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {(cuuint32_t)TILE_K, box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

// The same matrix for SMALL launches: box = two 64-column blocks of box_rows rows, one block behind the other (a last block
// that does not exist reads as zero).
inline CUresult encode_2d_small(EncodeTiledFn fn, CUtensorMap *tm, const void *base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  cuuint64_t dims[3] = {(cuuint64_t)TILE_K, rows, cols / TILE_K};
  cuuint64_t strides[2] = {cols * 2, TILE_K * 2};
  cuuint32_t box[3] = {(cuuint32_t)TILE_K, box_rows, (cuuint32_t)k_per_stage(true)};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

// Row-block geometry for R activation rows in n_rb blocks.
inline void plan_rows(int R, Args &a, int n_rb) {
  a.n_rb = n_rb;
  const int per = (R + n_rb - 1) / n_rb;
  a.rb_rows = (per + 15) / 16 * 16;
  a.n1 = a.rb_rows; a.n2 = 0;
  if (a.rb_rows > 256) { a.n1 = ((a.rb_rows / 2 + 15) / 16) * 16; a.n2 = a.rb_rows - a.n1; }
}
inline int stage_bytes(const Args &a, bool small) { return k_per_stage(small) * (W_STAGE_BYTES + (small ? a.rb_rows : a.rb_rows / 2) * TILE_K * 2); }
// Depth of the ring of a launch whose CTAs read n stages each.  A SMALL launch takes no more than n (the next projection's
// CTA may then sit on the same SM) and at most five (24 MB of weights in flight over the machine; the 8B-class step of
// 20 rows takes 4.0 ms with five, 4.05 with four, 4.5 with two and a half).
inline void plan_stages(Args &a, int n, bool small) {
  const int fit = SMEM_BUDGET / stage_bytes(a, small);
  a.stages = small ? std::max(2, std::min({5, fit, n})) : std::min(fit, MAX_STAGES);
}
inline size_t smem_bytes(const Args &a, bool small) { return (size_t)a.stages * stage_bytes(a, small) + 1024; }

// K splits of one row block: fill the workers (CTAs, or pairs) with whole waves of equally sized items, keeping at least
// min_kb stages per item; item_cost: fixed cost of an item in stages.
inline int plan_splits(int n_items_unsplit, int kb_total, int workers, int max_splits, int min_kb, double item_cost) {
  int best = 1; double best_eff = 0.0;
  for (int s = 1; s <= max_splits; ++s) {
    if (s > 1 && kb_total / s < min_kb) break;
    const long long items = (long long)n_items_unsplit * s;
    const long long waves = (items + workers - 1) / workers;
    const double eff = ((double)n_items_unsplit * kb_total) / ((double)waves * workers * ((double)((kb_total + s - 1) / s) + item_cost));
    if (eff > best_eff + 1e-9) { best_eff = eff; best = s; }
  }
  return best;
}
// The same for several row blocks, where slabs are large: blocks and split with the least estimated time.  Whole waves of items;
// per stage of K 2.15 cycles per row at 1.75 GHz; 1 us to hand an accumulator over; and S slabs of R x N floats written, and
// read again by the next kernel (max_splits = 0: no slabs, nothing is split).  Blocks take one instruction (up to 256 rows) or two (288):
// fewer blocks where that saves a wave.  (Chosen for whole waves alone, the O projection of 1152 rows was split 4 ways and a
// 4 k first pass spent 85 us per norm on slabs, 30 now.  1152 rows, 8B-class: O and its norm take 47 + 23 us as five blocks of 240 rows
// in two splits and 38 + 5.5 us as four of 288, unsplit; down and its norm 103 + 29 and 91 + 5.5 us.)
inline void plan_blocks(Args &a, int workers, int max_splits, int min_kb) {
  double best = 1e30;
  Args pick = a;
  for (int block : {BLOCK_ROWS, MAX_ROWS}) {
    plan_rows(a.R, a, (a.R + block - 1) / block);
    for (int S = 1; S == 1 || (S <= max_splits && a.kb_total / S >= min_kb); ++S) {
      const long long items = (long long)a.n_rb * a.n_tiles * S, waves = (items + workers - 1) / workers;
      const double us = (double)waves * (((a.kb_total + S - 1) / S) * ((2.15 * a.rb_rows + 50.0) / 1750.0) + 1.0) + (max_splits ? S * ((double)a.R * a.N * 6.0 / 5.0e6) : 0.0);
      if (us < best - 1e-9) { best = us; pick = a; pick.S = S; }
    }
  }
  a = pick;
}

}  // namespace gemm_tc
