// Structured-mask attention of one pass on tcgen05 tensor cores.
//
// A pass's rows (token slots) attend to the cached positions [0, nvis) of their sequence
// plus the nloc step-local K/V rows starting at loc0 (see RowMeta).  For a decode step this
// is the paper's decoding mask (figure "TiDAR Attention Masks"; Section 3.1): drafted
// tokens causal, every mask block bidirectional inside itself and blind to the other
// blocks.  The mask is never materialised: a query tile derives, from its rows' metadata,
// which 64-key pages it needs (cached pages up to the largest nvis, and only the local
// rows of the blocks it contains), skips all others, and applies the per-row bound only
// on pages that straddle it.
//
// Tiling: the G = Hq/Hkv query heads that share a KV head are packed into 128-row MMA tiles
// (floor(128/G) slots x G heads), so K/V are read once per KV head.  A CTA runs two streams, A and B, of
// (128-row query tile) x (64-key page) steps.  Per step j of stream T: S = Q_T K^T (M 128, N 64, K hd) into
// TMEM (double buffered); the stream's four softmax warps read S (one thread per row), keep a reference max
// and the running sum, and write P (bf16, two keys per 32-bit column) back over the first half of the
// S buffer it came from; O_T += P V (M 128, N hd, K 64, P as the tensor-memory operand, V as the MN-major
// shared-memory operand) accumulates in TMEM over all steps.  The streams take turns on the tensor pipe, and
// each has the scores of its next step waiting when it finishes one, so neither the pipe nor the softmax warps wait
// for the other's latency.
// What bounds it: shared memory.  A step's operands are 64 KB read (Q 32, K 16, V 16) and up to 32 KB written by
// the loads, 500 - 750 cycles at 128 B per cycle against 512 cycles of MMAs (a product with N = 64 takes 48 cycles, not
// 32, for the 6 KB it reads); a step takes 0.53 - 0.56 us, 0.93 - 0.98 kcycles, on an SM.  Whole calls with warm caches, 32/8
// heads of 128, 272 rows, 1 k / 4 k / 16 k / 32 k cached positions: 16.5 / 33 / 84 / 153 us; the kernel before this one
// (two CTAs per SM, one tile and one stream each, the same split for every sequence) took 26.2 / 40 / 97 / 173 us.
//   PAIR of tiles: A and B are two query tiles, each K/V page serves both: half the loads, and 80
//     instead of 96 KB through shared memory per step.
//   SINGLE tile: A and B are the same query tile and take the pages in turn; their two results are merged through
//     shared memory at the end.  Twice the parallelism for the same rows and half the partial results.
//
// One thread issues all MMAs, and a commit covers everything issued before it: the barrier that announces
// the scores of step j + 2 (their products are issued right behind P V of step j, and the barrier is committed
// to even when there are no such scores) also says that P V of step j has read its P and updated O.
// The reference max is only raised when a step exceeds it by more than 2^8 (P stays <= 256,
// exact enough in bf16/fp32); raising it rescales the rows of O in TMEM, which happens in the
// first steps only.
//
// As in the projections, the thread that issues MMAs never tests an mbarrier (the test would wait for the MMAs
// queued before it and the pipe would run dry): a watcher warp does, and releases it through
// hardware barriers.
//
// Work distribution.  Which CTA does what is planned on the device, once per pass (plan_block):
// every layer of a pass has the same rows, hence the same query tiles and key ranges.  The plan decides whether
// tiles are paired, cuts key ranges into items of about equal time, whatever the sequences' lengths
// are, and lists long items first (a causal first pass would otherwise end on its longest rows).
// Partial (max, sum, O) results of a tile with several items are merged by attn_combine_kernel.
// A stand-alone call pays for its plan alone (4.5 us).  Where there is little to distribute it does without: every CTA
// works out its own item (direct_item), with an instance of one stream per CTA where that saves a wave.
#pragma once
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace attn_tc {

constexpr int PAGE = 64;             // keys per step (= page size)
// warp 0: K loads, 1: MMA, 2: watcher, 3: Q and V loads; warps 4..7 / 8..11: softmax of stream A / B
__host__ __device__ constexpr int threads(int streams) { return 128 + 128 * streams; }
constexpr int MAX_SPLITS = 32;       // items per tile
constexpr int MAX_CLUSTER = 8;       // CTAs that may share an item
constexpr int SLOTS_PER_SM = 2;      // partial results that fit the scratch = grid of a pass whose key ranges may be split
constexpr float RAISE_THRESHOLD = 8.f;   // log2 units

// Pages [p_begin, p_end) of the query tile that covers slots [row0, min(row0 + spt, row_end)) of sequence slot `seq`
// and, if pair, of the tile behind it.  Its keys in pages: n_cache_pages cached ones, then step-local rows from loc_lo on.
struct __align__(16) Item { int32_t row0, row_end, seq, p_begin, p_end, n_cache_pages, loc_lo, pair, split, pad[3]; };
// A query tile: its items are item0 .. item0 + n_items - 1 (n_items = 0: no rows); in a pair, sub says which half it is.
struct __align__(16) Tile { int32_t row0, row_end, item0, n_items, sub, pad[3]; };

// Units (up to two query tiles of one sequence) of a pass and where the plan goes.
struct PlanArgs {
  int R;                    // rows (slots) of the pass
  int rows_per_group;       // slots per sequence group (k(k+1) for a step; R for a first pass)
  int units_per_group;      // ceil(rows_per_group / (2 spt))
  // Groups of different sizes (a step whose sequences use different block lengths): unit u
  // covers rows [unit_row0[u], unit_row0[u] + 2 spt) of the group that ends at unit_rend[u]; null =
  // equal groups, derived from rows_per_group.  n_units = number of units in either case.
  const int32_t *unit_row0, *unit_rend; int n_units;
  int spt;                  // slots per query tile = 128 / G
  int Hkv;
  int n_sms, max_items;     // items a pass may have; n_units = every unit is one item
  int max_pieces;           // items a tile or pair may have (1: nothing is split, the merge kernel is not launched)
  int singles;              // tiles are not paired (an item is shared by a cluster, see attn_tc_kernel)
  Item *items; Tile *tiles; // out: [max_items] (unused ones are zero), [2 n_units] (only where items may be split)
};

struct Args {
  int spt;                  // slots per query tile = 128 / G
  int G, Hq, Hkv;
  const Item *items; const Tile *tiles;
  const int32_t *nvis, *loc0, *nloc;         // per row
  const int32_t *page_table; int pages_per_seq;
  int page_base_k, page_base_v;              // offsets in the page dimension of the K / V tensor maps
  float scale_log2;                          // log2(e) / sqrt(hd)
  bf16 *O;                                   // [R][Hq*hd]
  float *part_O;                             // [CTA][tile of the pair][hd / 4][128 rows][4]: a warp's stores are contiguous
  float2 *part_ml;                           // [CTA][tile of the pair][128 rows] (reference max, sum)
  // early: plan, row metadata and page table, which were written before the pass's first RoPE kernel, are read ahead of pdl_wait(): that kernel
  // lets its successor in only once its own predecessors are complete, and every later kernel of the pass starts after that
  int early;
  // Stand-alone calls without a plan (items = null; DIRECT instances): what a CTA works out its item and its rows' keys from.
  struct { const int32_t *seq_len; int k, n_max; int per_group, pieces; } direct;    // query tiles per sequence, items per tile at most
  int *status;
  unsigned long long *tile_count;            // diagnostics: += steps this CTA computes (null = off)
};

// Shared memory of one CTA; everything is dynamic so that the 1024-byte alignment the
// swizzled tiles need costs no padding (the kernel checks the base address).
template <int HD, int STREAMS = 2, bool CLUSTER = false>
struct Smem {
  static constexpr int K_STAGES = CLUSTER ? 4 : STREAMS == 2 ? 5 : 3, V_STAGES = CLUSTER ? 3 : STREAMS == 2 ? 5 : 2;     // pages in flight (one stream: two CTAs fit an SM)
  static constexpr int NH = HD / 64;                 // 64-element halves of a head
  static constexpr int Q_BYTES = 128 * HD * 2;       // one query tile
  static constexpr int KV_BYTES = PAGE * HD * 2;
  static constexpr int Q_OFF = 0;
  static constexpr int K_OFF = Q_OFF + (CLUSTER ? 1 : STREAMS) * Q_BYTES;
  static constexpr int V_OFF = K_OFF + K_STAGES * KV_BYTES;
  // CLUSTER: this CTA's columns of the tile's result as every CTA of the cluster has them, [CTA][stream][columns / 4][128 rows][4] floats, and
  // the CTAs' (reference max, sum), [CTA][128 rows].  (Written by the others at any time, hence a place of its own.)
  static constexpr int PEER_OFF = V_OFF + V_STAGES * KV_BYTES, PEER_ML_OFF = PEER_OFF + (CLUSTER ? 128 * HD * 4 : 0);
  static constexpr int BAR_OFF = PEER_ML_OFF + (CLUSTER ? MAX_CLUSTER * 128 * 8 : 0);    // mbarriers and a few words
  static constexpr int TOTAL = BAR_OFF + 512;
  static constexpr int XCHG_OFF = K_OFF;             // single tile: the streams' results, [stream][hd / 8][128 rows][4] floats; (max, sum) behind them
  static constexpr int XCHG_ML_OFF = XCHG_OFF + 128 * HD * 4;
  static constexpr int TMEM_COLS = 256 * STREAMS;    // per stream 2 x 64 (S) + HD (O), rounded up to a power of two
};
static_assert(Smem<128, 2, true>::XCHG_ML_OFF + 2 * 128 * 8 <= Smem<128, 2, true>::PEER_OFF && Smem<64, 2, true>::XCHG_ML_OFF + 2 * 128 * 8 <= Smem<64, 2, true>::PEER_OFF &&
              Smem<128, 2, true>::TOTAL <= 227 * 1024, "exchange area fits the K/V rings of a cluster's CTA");
static_assert(Smem<128>::XCHG_ML_OFF + 2 * 128 * 8 <= Smem<128>::BAR_OFF && Smem<64>::XCHG_ML_OFF + 2 * 128 * 8 <= Smem<64>::BAR_OFF, "exchange area fits the K/V rings");

struct Ctl {                                         // lives at Smem::BAR_OFF
  uint64_t q_full, k_full[5], k_empty[5], v_full[5], v_empty[5], s_full[2][2], p_full[2][2];
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(Ctl) <= 512, "control block must fit its slot");

// Plans a pass's attention (see the head of this file); run by one whole block, a multiple of 128 threads.
//
// The entities of a plan are the units (tiles paired) or the tiles (not paired).  Every entity's key range is cut
// into the fewest items of at most `limit` us.  Pairing and limit minimise an estimate of
// the kernel's time: a CTA costs OVERHEAD us (first loads, first scores, result) and per page PAIR_PAGE or
// SINGLE_PAGE us; a partial result costs its store (PAIR_STORE, SINGLE_STORE) and the merge kernel; CTAs beyond one per
// SM run in later waves, of which on average half a CTA's time is lost at the end.
// Everything is kept in shared memory until the plan is made: a trip to global memory and back costs as much as all
// of the arithmetic.
// (Measured inside the kernel, head_dim 128, all SMs busy: 1.05 us per page of a pair, 0.56 of a single tile.  head_dim 64 and nearly empty
// grids take the same figures, although a page costs them less: they were not fitted, and cuts come out somewhat finer than best.)
constexpr float CLUSTER_MERGE = 2.f;                   // what sharing an item within a cluster adds
// A stand-alone call is launched in clusters for the width of its page table, which is all the host knows; a tile whose own pages (known on the device) are
// few is its cluster's first CTA's alone.  Shared where that takes at least CLUSTER_SAVES pages off the longest CTA (four SINGLE_PAGE: what sharing costs).
// Alone / shared, tables of 8 to 16 pages: 32/8 heads of 128, k = 4, clusters of eight, 2 pages per tile 7.2 / 8.1 us, 5 pages 7.9 / 8.4, 6 pages 8.9 / 8.4;
// 12/2 heads, k = 16, clusters of four, 2 pages 8.0 / 9.8, 5 pages 9.9 / 10.2, 6 pages 10.4 / 10.3; 4/2 heads of 64, k = 4, 6 pages 7.7 / 6.9.  (A step's sizes
// are known on the host.)
constexpr int CLUSTER_SAVES = 4;
__host__ __device__ constexpr bool cluster_shares(int n_pages, int log_size) { return n_pages - ((n_pages + (1 << log_size) - 1) >> log_size) >= CLUSTER_SAVES; }
constexpr float OVERHEAD = 5.f, PAIR_PAGE = 1.05f, SINGLE_PAGE = 0.56f, PAIR_STORE = 2.5f, SINGLE_STORE = 1.5f, MERGE = 3.f;
constexpr int PLAN_UNITS = 256;                        // up to this many units are planned; beyond, every unit is one item
constexpr int CAND = 32;                               // limits tried per pairing: longest / (1 + i / 2)

// The estimate, for the plan kernel and for the host, which decides with it whether a step's merge kernel is needed at all (step_attention): limit number i
// of the units or tiles the longest of which takes `longest` us; pieces of an entity of `us` us, at most one per page; what all entities come to.
struct PlanCost { int items, live, most; float sum, longest; };
__host__ __device__ inline float plan_limit(float longest, int i) { return fmaxf(longest / (1.f + 0.5f * i), 0.1f) * 1.0001f; }
__host__ __device__ inline int plan_pieces(float us, float limit, bool dbl) {
  const float n = us / limit, pages = us * (dbl ? 1.0001f / PAIR_PAGE : 1.0001f / SINGLE_PAGE);
#ifdef __CUDA_ARCH__
  return (int)fminf(ceilf(n), pages);
#else
  const int up = (int)n + ((float)(int)n < n ? 1 : 0);           // (the same without a library call)
  return std::min(up, (int)pages);
#endif
}
__host__ __device__ inline void plan_add(PlanCost &c, float us, float limit, bool dbl, int times = 1) {
  const int k = plan_pieces(us, limit, dbl);
  const float store = k > 1 ? (dbl ? PAIR_STORE : SINGLE_STORE) : 0.f;
#ifdef __CUDA_ARCH__
  const float piece = __fdividef(us, (float)k);
#else
  const float piece = us / (float)k;
#endif
  c.items += times * k; c.live += times; c.most = k > c.most ? k : c.most;
  c.sum += times * (us + k * (OVERHEAD + store));
  c.longest = fmaxf(c.longest, piece + (k > 1 ? 0.5f * SINGLE_PAGE : 0.f) + store + OVERHEAD);
}
__host__ __device__ inline float plan_time(const PlanCost &c, int Hkv, int n_sms) {
  float us = c.longest;
  if (c.items * Hkv > n_sms) us = fmaxf(us, Hkv * c.sum / n_sms + 0.5f * c.longest);
  if (c.items > c.live) us += MERGE + 0.3f * c.items / c.live;
  return us;
}

// What a row sees: cached positions [0, nvis), local rows [loc0, loc0 + nloc).
struct RowKeys { int nvis, loc0, nloc, seq; };

template <typename ROW>
__device__ inline void plan_block(const PlanArgs &p, ROW row_keys) {
  struct Keys { int n_cache, n_pages, loc_lo; };       // (a sequence of more than 32767 pages fits a B200)
  __shared__ Keys keys[3][PLAN_UNITS];                 // tile 0, tile 1, the unit
  __shared__ int unit_row0[PLAN_UNITS], unit_rend[PLAN_UNITS], unit_seq[PLAN_UNITS];
  __shared__ float ent_us[3 * PLAN_UNITS];             // units, then tiles
  __shared__ short ent_n[2 * PLAN_UNITS], order_s[2 * PLAN_UNITS], place_s[2 * PLAN_UNITS];
  __shared__ int longest_us[2];                        // longest unit / tile, as float bits
  __shared__ unsigned long long best[32];              // per warp (64-bit atomics in shared memory would take turns)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  const bool planned = p.n_units <= PLAN_UNITS, splits = p.max_items > p.n_units;
  if (threadIdx.x < 2) longest_us[threadIdx.x] = 0;
  __syncthreads();
  for (int u = warp; u < p.n_units; u += n_warps) {
    int row0, row_end;
    if (p.unit_row0) { row0 = p.unit_row0[u]; row_end = p.unit_rend[u]; }
    else {
      const int i = u % p.units_per_group, grp = u / p.units_per_group;
      row0 = grp * p.rows_per_group + i * 2 * p.spt;
      row_end = min((grp + 1) * p.rows_per_group, p.R);
    }
    int nvis[2] = {0, 0}, lo[2] = {0x7fffffff, 0x7fffffff}, hi[2] = {0, 0}, seq = 0;
    for (int r = row0 + lane; r < min(row0 + 2 * p.spt, row_end); r += 32) {
      const RowKeys k = row_keys(r);
      const int t = r >= row0 + p.spt;
      seq = k.seq;
      if (t) { nvis[1] = max(nvis[1], k.nvis); if (k.nloc > 0) { lo[1] = min(lo[1], k.loc0); hi[1] = max(hi[1], k.loc0 + k.nloc); } }
      else { nvis[0] = max(nvis[0], k.nvis); if (k.nloc > 0) { lo[0] = min(lo[0], k.loc0); hi[0] = max(hi[0], k.loc0 + k.nloc); } }
    }
    seq = __shfl_sync(0xffffffffu, seq, 0);            // (row0 itself is lane 0's)
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      nvis[t] = __reduce_max_sync(0xffffffffu, nvis[t]); lo[t] = __reduce_min_sync(0xffffffffu, lo[t]); hi[t] = __reduce_max_sync(0xffffffffu, hi[t]);
    }
    if (lane < 3) {                                    // lane 0 / 1: the tiles, lane 2: the unit
      const int nv = lane == 0 ? nvis[0] : lane == 1 ? nvis[1] : max(nvis[0], nvis[1]);
      const int l = lane == 0 ? lo[0] : lane == 1 ? lo[1] : min(lo[0], lo[1]), h = lane == 0 ? hi[0] : lane == 1 ? hi[1] : max(hi[0], hi[1]);
      const bool two = row0 + p.spt < row_end;
      const int n_cache = (nv + PAGE - 1) / PAGE, n_pages = n_cache + (h > l ? (h - l + PAGE - 1) / PAGE : 0);
      if (planned) {
        keys[lane][u] = Keys{n_cache, n_pages, l};
        const float us = n_pages * (lane == 2 && two ? PAIR_PAGE : SINGLE_PAGE);
        ent_us[lane == 2 ? u : p.n_units + 2 * u + lane] = us;
        atomicMax(&longest_us[lane == 2 ? 0 : 1], __float_as_int(us));
        if (lane == 0) { unit_row0[u] = row0; unit_rend[u] = row_end; unit_seq[u] = seq; }
      } else if (lane == 2) {                          // every unit one item, listed back to front (a causal pass lists its rows in ascending length)
        Item it{};
        it.row0 = row0; it.row_end = row_end; it.seq = seq; it.p_end = n_pages; it.n_cache_pages = n_cache; it.loc_lo = l; it.pair = two;
        p.items[p.n_units - 1 - u] = it;
      }
    }
  }
  if (!planned) return;
  __syncthreads();
  bool paired = true;
  float limit = 1e30f;
  auto limit_of = [&](int cnd) { return plan_limit(__int_as_float(longest_us[cnd / CAND]), cnd % CAND); };
  if (splits) {
    const int per = blockDim.x / (2 * CAND) >= 16 ? 16 : blockDim.x / (2 * CAND) >= 4 ? 4 : 2;       // threads per candidate
    const int cnd = threadIdx.x / per, sub = threadIdx.x % per;
    const bool live_cnd = cnd < 2 * CAND, pr = cnd < CAND;
    const float lim = limit_of(live_cnd ? cnd : 0);
    const int n_ent = live_cnd ? (pr ? p.n_units : 2 * p.n_units) : 0, e0 = pr ? 0 : p.n_units;
    PlanCost cost{0, 0, 0, 0.f, 0.f};
    for (int e = sub; e < n_ent; e += per) {
      const float us = ent_us[e0 + e];
      if (us > 0.f) plan_add(cost, us, lim, pr && unit_row0[e] + p.spt < unit_rend[e]);
    }
    for (int o = per >> 1; o > 0; o >>= 1) {
      cost.items += __shfl_xor_sync(0xffffffffu, cost.items, o); cost.live += __shfl_xor_sync(0xffffffffu, cost.live, o);
      cost.most = max(cost.most, __shfl_xor_sync(0xffffffffu, cost.most, o));
      cost.sum += __shfl_xor_sync(0xffffffffu, cost.sum, o); cost.longest = fmaxf(cost.longest, __shfl_xor_sync(0xffffffffu, cost.longest, o));
    }
    unsigned long long mine = ~0ull;
    if (live_cnd && cost.items <= p.max_items && cost.most <= p.max_pieces && !(pr && p.singles))
      mine = ((unsigned long long)__float_as_uint(plan_time(cost, p.Hkv, p.n_sms)) << 32) | (unsigned)cnd;      // (positive: its bits order like its value)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine = min(mine, __shfl_xor_sync(0xffffffffu, mine, o));
    if (lane == 0) best[warp] = mine;
    __syncthreads();
    mine = lane < n_warps ? best[lane] : ~0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine = min(mine, __shfl_xor_sync(0xffffffffu, mine, o));
    if (mine != ~0ull) { const int c = (int)(mine & 0xffffffffu); paired = c < CAND; limit = limit_of(c); }
  }
  const int n_ent = paired ? p.n_units : 2 * p.n_units, e0 = paired ? 0 : p.n_units;
  for (int e = threadIdx.x; e < n_ent; e += blockDim.x) {
    const float us = ent_us[e0 + e];
    const int k = us <= 0.f ? 0 : splits ? max(1, plan_pieces(us, limit, paired && unit_row0[e] + p.spt < unit_rend[e])) : 1;
    ent_n[e] = (short)k; ent_us[e0 + e] = k ? us / k : -1.f;
  }
  __syncthreads();
  // longest items first: entity e goes to place `rank`
  for (int e = threadIdx.x; e < n_ent; e += blockDim.x) {
    const float us = ent_us[e0 + e];
    int rank = 0;
#pragma unroll 4
    for (int f = 0; f < n_ent; ++f) { const float v = ent_us[e0 + f]; rank += v > us || (v == us && f < e); }
    order_s[rank] = (short)e;
  }
  __syncthreads();
  if (warp == 0) {                                     // places of the items: running sum over the order
    int base = 0;
    for (int r0 = 0; r0 < n_ent; r0 += 32) {
      const int e = r0 + lane < n_ent ? order_s[r0 + lane] : -1;
      const int n = e >= 0 ? ent_n[e] : 0;
      int sum = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, sum, o); if (lane >= o) sum += v; }
      if (e >= 0) place_s[e] = (short)(base + sum - n);
      base += __shfl_sync(0xffffffffu, sum, 31);
    }
    for (int i = base + lane; i < p.max_items; i += 32) p.items[i] = Item{};       // unused places: no rows, no pages
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 2 * p.n_units; t += blockDim.x) {                  // what the merge kernel needs
    const int u = t >> 1, e = paired ? u : t;
    Tile w{};
    w.row0 = unit_row0[u] + (t & 1) * p.spt; w.row_end = unit_rend[u];
    w.n_items = w.row0 < w.row_end ? ent_n[e] : 0; w.item0 = place_s[e]; w.sub = paired ? t & 1 : 0;
    p.tiles[t] = w;
  }
  for (int e = warp; e < n_ent; e += n_warps) {
    const int u = paired ? e : e >> 1, n = ent_n[e];
    const Keys k = keys[paired ? 2 : e & 1][u];
    for (int j = lane; j < n; j += 32) {
      Item it{};
      it.row0 = unit_row0[u] + (paired ? 0 : (e & 1) * p.spt); it.row_end = unit_rend[u]; it.seq = unit_seq[u];
      it.n_cache_pages = k.n_cache; it.loc_lo = k.loc_lo;
      it.p_begin = k.n_pages * j / n; it.p_end = k.n_pages * (j + 1) / n;      // (2^31 positions are 2^25 pages, in at most 2^5 pieces)
      it.pair = paired && unit_row0[u] + p.spt < unit_rend[u]; it.split = n > 1;
      p.items[place_s[e] + j] = it;
    }
  }
}

// What row r of a stand-alone call sees (the slot layout of a step of equal block lengths k).  seq_len comes from the caller: it is
// clamped to [0, n_max] (the positions the page table can back minus the k causal slots), so that no row looks past the table.
__device__ __forceinline__ RowKeys step_row_keys(const int32_t *__restrict__ seq_len, int k, int n_max, int r) {
  const int T = k * (k + 1);
  const int s = r / T, slot = r % T;
  const int n = min(max(seq_len[s], 0), n_max);
  if (slot < k) return RowKeys{n + slot + 1, 0, 0, s};
  const int b = (slot - k) / k;
  return RowKeys{n + b + 1, s * k * k + b * k, k, s};
}

// Query tile number `tile` of a stand-alone call that has no plan, with its whole key range, as an item.
__device__ __forceinline__ Item direct_tile(const Args &a, int tile) {
  const int k = a.direct.k, T = k * (k + 1), s = tile / a.direct.per_group, first = tile % a.direct.per_group * a.spt;
  const int last = min(first + a.spt, T) - 1;                    // its slots
  // the causal slots see more the later they come, the mask blocks too, and the last causal slot sees what the last block sees
  const RowKeys most = step_row_keys(a.direct.seq_len, k, a.direct.n_max, s * T + (first < k ? min(last, k - 1) : last));
  Item it{};
  it.row0 = s * T + first; it.row_end = (s + 1) * T; it.seq = s;
  it.p_end = it.n_cache_pages = (most.nvis + PAGE - 1) / PAGE;
  if (last >= k) {
    it.loc_lo = s * k * k + (max(first, k) - k) / k * k;
    it.p_end += (s * k * k + ((last - k) / k + 1) * k - it.loc_lo + PAGE - 1) / PAGE;
  }
  return it;
}
// Items that a tile of n_pages pages is cut into (three pages at least: see attention_direct), out of the places it has.
__device__ __forceinline__ int direct_pieces(const Args &a, int n_pages) { return max(1, min(a.direct.pieces, n_pages / 3)); }
__device__ __forceinline__ Item direct_item(const Args &a, int e) {
  Item it = direct_tile(a, e / a.direct.pieces);
  const int j = e % a.direct.pieces, n = direct_pieces(a, it.p_end), n_pages = it.p_end;
  it.split = n > 1;
  it.p_begin = j < n ? n_pages * j / n : 0; it.p_end = j < n ? n_pages * (j + 1) / n : 0;      // a place that is not used has no pages
  return it;
}

// The end of a tile that its cluster does not share: both streams' halves merged and written.  A function of its own, called, so that its code does not
// lie in the way of shared tiles (in place it cost them 0.1 - 0.2 us, as branches in their loop 0.3).
template <int HD>
__device__ __noinline__ void finish_alone(uint32_t o_addr, int t, int my_row, float m_ref, float l_run, int nj, bf16 *o, const float4 *xo, const float2 *xml) {
  const float2 other = xml[(1 - t) * 128 + my_row];
  const float M = fmaxf(m_ref, other.x);
  const float wm = m_ref == -INFINITY ? 0.f : exp2f(m_ref - M), wo = other.x == -INFINITY ? 0.f : exp2f(other.x - M);
  const float inv = 1.f / (wm * l_run + wo * other.y);
#pragma unroll 1
  for (int c = 0; c < HD / 2; c += 32) {
    uint32_t w[32];
    float v[32];
    if (nj > 0) { sm100::tmem_ld32(o_addr + t * (HD / 2) + c, w); sm100::tmem_wait_ld(); }
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = nj > 0 ? __uint_as_float(w[i]) : 0.f;
#pragma unroll
    for (int i = 0; i < 32; i += 4) {
      const float4 x = xo[(t * (HD / 8) + (c + i) / 4) * 128 + my_row];
      v[i] = wm * v[i] + wo * x.x; v[i + 1] = wm * v[i + 1] + wo * x.y; v[i + 2] = wm * v[i + 2] + wo * x.z; v[i + 3] = wm * v[i + 3] + wo * x.w;
    }
    if (o) {
#pragma unroll
      for (int i = 0; i < 32; i += 8) {
        uint4 u;
        __nv_bfloat162 h0 = __floats2bfloat162_rn(v[i] * inv, v[i + 1] * inv), h1 = __floats2bfloat162_rn(v[i + 2] * inv, v[i + 3] * inv),
                       h2 = __floats2bfloat162_rn(v[i + 4] * inv, v[i + 5] * inv), h3 = __floats2bfloat162_rn(v[i + 6] * inv, v[i + 7] * inv);
        u.x = *reinterpret_cast<uint32_t *>(&h0); u.y = *reinterpret_cast<uint32_t *>(&h1);
        u.z = *reinterpret_cast<uint32_t *>(&h2); u.w = *reinterpret_cast<uint32_t *>(&h3);
        *reinterpret_cast<uint4 *>(o + t * (HD / 2) + c + i) = u;
      }
    }
  }
}

// STREAMS = 1: one tile and one stream per CTA and two CTAs per SM, which fill each other's latencies as two streams do.  It serves calls that are
// one wave that way and two otherwise (see attention_direct for both sides' figures).  DIRECT: no plan, see direct_item.
// AHEAD (decode steps of few rows, whose CTAs become resident well before the RoPE kernel ends): what does not depend on that kernel is done ahead of
// the wait.  The rows of a step see at most 64 positions more than their sequence had cached before it, so of n cached pages a query tile
// needs, no kernel of the step writes the first n - 2, and those go into the rings at once; they come from HBM, the weights of a step having passed
// through the L2 since the last one.  And the softmax warps walk through one step with nothing stored, on whatever tensor memory holds, which
// fetches the loop's code.  (8B-class step of 20 rows: 10.1 us behind a gap of 0.77 -> 8.9 behind 0.70; 1.5B-class autoregressive step of 8 rows 6.05 -> 4.75.
// At 272 rows the CTAs wait for the SMs of the projection in front of the RoPE kernel and only lose by it; walking through the output code too was slower
// everywhere, by 0.8 - 2 us.)
// CLUSTER: the CTAs of a cluster share an item (a single tile, not cut; of a stand-alone call only one of enough pages, see cluster_shares): each takes an
// even share of its pages, and their results are merged over
// distributed shared memory: every CTA finishes 1 / size of the head's columns, which the others store into its shared memory.  For calls and steps of few
// tiles and contexts of some pages (see attention_direct, step_attention); bound by the latencies of first load and merge, about 2 us for the latter
// (CLUSTER_MERGE).  Alone, 32/8 heads of 128, 272 rows, 1 k positions, clusters of two: 15.8 -> 13.2 us; 12/2 heads, four sequences of 72 rows, 1 k
// positions, clusters of four: 16.5 -> 11.7.  1.5B-class step of 272 rows: 10.4 -> 8.1 us per layer; autoregressive step of 8 rows, where it replaces
// a cut and the merge kernel: 5.1 + 3.4 -> 7.5 us.
template <int HD, int STREAMS, bool DIRECT, bool AHEAD, bool CLUSTER>
__global__ void __launch_bounds__(threads(STREAMS), 3 - STREAMS)
attn_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
               const __grid_constant__ CUtensorMap tmKloc, const __grid_constant__ CUtensorMap tmVloc, const Args a, const TlSlot tl) {
  using L = Smem<HD, STREAMS, CLUSTER>;
  constexpr int NH = L::NH;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const int warp = sm100::warp_index(), lane = threadIdx.x & 31;
  const uint32_t smem0 = sm100::smem_u32(smem_raw);
  if (smem0 & 1023u) {                               // cannot place swizzled tiles: report, touch nothing
    if (threadIdx.x == 0 && a.status) atomicExch(a.status, 3);
    return;
  }
  Ctl &ctl = *reinterpret_cast<Ctl *>(smem_raw + L::BAR_OFF);
  const int rows_used = a.spt * a.G;                                   // MMA rows of a tile that carry data

  if (warp == 2 && lane < 5) sm100::prefetch_tensormap(lane == 0 ? &tmQ : lane == 1 ? &tmK : lane == 2 ? &tmV : lane == 3 ? &tmKloc : &tmVloc);
  if (threadIdx.x == 0) {
    ctl.abort_flag = 0;
    sm100::mbar_init(sm100::smem_u32(&ctl.q_full), 1);
    for (int s = 0; s < L::K_STAGES; ++s) { sm100::mbar_init(sm100::smem_u32(&ctl.k_full[s]), 1); sm100::mbar_init(sm100::smem_u32(&ctl.k_empty[s]), 1); }
    for (int s = 0; s < L::V_STAGES; ++s) { sm100::mbar_init(sm100::smem_u32(&ctl.v_full[s]), 1); sm100::mbar_init(sm100::smem_u32(&ctl.v_empty[s]), 1); }
    for (int t = 0; t < STREAMS; ++t)
      for (int b = 0; b < 2; ++b) { sm100::mbar_init(sm100::smem_u32(&ctl.s_full[t][b]), 1); sm100::mbar_init(sm100::smem_u32(&ctl.p_full[t][b]), 4); }
    sm100::fence_mbar_init();
  }
  if (warp == 1) {
    __syncwarp();
    sm100::tmem_alloc(sm100::smem_u32(&ctl.tmem_base), L::TMEM_COLS);
    sm100::tmem_relinquish();
  }
  sm100::tc_fence_before();
  __syncthreads();
  sm100::tc_fence_after();
  if constexpr (CLUSTER) sm100::cluster_arrive_relaxed();     // this CTA runs (waited for before the first store to another one)
  const uint32_t tmem = ctl.tmem_base;
  const uint32_t tmem_S = tmem, tmem_O = tmem + STREAMS * 2 * PAGE;   // per stream: 2 x 64 columns of S, HD columns of O
  volatile int *abortp = &ctl.abort_flag;
  pdl_trigger();              // not before the tensor memory is ours (see gemm_tc_kernel)
  if (DIRECT || !a.early) pdl_wait();

  // ---- which work item (every thread reads it: no barrier before the first loads go out) ----
  const int c_size = CLUSTER ? (int)sm100::cluster_size() : 1, c_rank = CLUSTER ? (int)sm100::cluster_rank() : 0;
  const int c_log = 31 - __clz(c_size);                // (a power of two: shifts instead of divisions ahead of the first loads, 0.1 us)
  const int kvh = (blockIdx.x >> c_log) % a.Hkv, item_no = (blockIdx.x >> c_log) / a.Hkv;
  Item item = DIRECT ? direct_item(a, item_no) : a.items[item_no];   // all zero where the grid is larger than the plan: nothing to do
  const int np_item = item.p_end - item.p_begin;
  const bool sharing = CLUSTER && (!DIRECT || cluster_shares(np_item, c_log));     // (the same in all CTAs of a cluster)
  if constexpr (CLUSTER) {
    const int b = item.p_begin;
    if (sharing) { item.p_begin = b + (np_item * c_rank >> c_log); item.p_end = b + (np_item * (c_rank + 1) >> c_log); }
    else if (c_rank > 0) item.p_end = b;
  }
  const int row0 = item.row0, p_begin = item.p_begin, np = item.p_end - item.p_begin;
  const bool pair = STREAMS == 2 && !CLUSTER && item.pair != 0;
  const bool shared = STREAMS == 1 || pair;                            // every stream takes every page; otherwise two streams take them in turn
  const int ahead = shared ? 2 : 4;                                    // pages whose scores are computed ahead: two steps of every stream
  auto stream0 = [&](int p) { return shared ? 0 : p & 1; };            // streams [stream0(p), stream1(p)) take page p
  auto stream1 = [&](int p) { return pair ? 2 : stream0(p) + 1; };
  if (threadIdx.x == 0 && a.tile_count && np > 0) atomicAdd(a.tile_count, (unsigned long long)np * (pair ? 2 : 1));

  const int t = (warp - 4) >> 2;                         // softmax warps: stream
  const int my_row = (warp & 3) * 32 + lane;             // and this thread's MMA row = TMEM lane
  int my_slot = -1;                                      // and its slot, -1: none
  const int c_cols = (HD / 2) >> c_log, c_shift = 31 - __clz(c_cols);     // columns of a stream's half that a CTA of the cluster finishes (at least 8)
  if (warp == 0 || warp == 3) {
    // ===================== K producer / Q and V producer =====================
    // Lane i holds the i-th entry of a group of 32 entries of the page table, so that a page's load does not wait for
    // its entry.  One load per page (the halves of the head are a dimension of the tensor map), and K and V each have
    // a warp of their own: issuing a page's four loads one after the other from one warp took 1700 cycles per
    // page (of 64 keys), three times as long as the page's MMAs.
    if (np > 0) {
      const bool is_k = warp == 0;
      const uint64_t pol = sm100::policy_evict_last();
      const int32_t *table = a.page_table + (size_t)item.seq * a.pages_per_seq;
      const int n_table = min(item.n_cache_pages, item.p_end) - p_begin;         // pages of this item that the table backs
      int cur = lane < n_table ? table[p_begin + lane] : 0, next = 0;
      const CUtensorMap *tm = is_k ? &tmK : &tmV, *tm_loc = is_k ? &tmKloc : &tmVloc;
      const int base = is_k ? a.page_base_k : a.page_base_v;
      const int stages = is_k ? L::K_STAGES : L::V_STAGES;
      const uint32_t full0 = sm100::smem_u32(is_k ? ctl.k_full : ctl.v_full), empty0 = sm100::smem_u32(is_k ? ctl.k_empty : ctl.v_empty);
      const uint32_t dst0 = smem0 + (is_k ? L::K_OFF : L::V_OFF);
      const int n_ahead = AHEAD ? max(min(min(item.n_cache_pages - 2 - p_begin, np), stages), 0) : 0;
      int s = 0; uint32_t ph = 1u;
      for (int p = 0;; ++p) {
        if (p == n_ahead) {
          pdl_wait();                                  // Q and all other pages are the previous kernel's output
          if (threadIdx.x == 0) tl_go(tl);
          if (!is_k && sm100::elect_one()) {
            const uint32_t qb = sm100::smem_u32(&ctl.q_full);
            sm100::mbar_expect_tx(qb, (uint32_t)(NH * rows_used * 128 * (pair ? 2 : 1)));
            for (int t = 0; t < (pair ? 2 : 1); ++t)
              for (int h = 0; h < NH; ++h)
                sm100::tma_load_3d(smem0 + L::Q_OFF + t * L::Q_BYTES + h * (128 * 128), &tmQ, qb, h * 64, kvh * a.G, row0 + t * a.spt, pol);
          }
          __syncwarp();
        }
        if (p == np) break;
        if ((p & 31) == 0) {
          if (p) cur = next;
          next = p + 32 + lane < n_table ? table[p_begin + p + 32 + lane] : 0;
        }
        const int page = __shfl_sync(0xffffffffu, cur, p & 31) + base;
        if (!sm100::mbar_wait_warp(empty0 + (uint32_t)s * 8u, ph, abortp)) break;
        if (sm100::elect_one()) {
          const uint32_t fb = full0 + (uint32_t)s * 8u, dst = dst0 + (uint32_t)s * L::KV_BYTES;
          sm100::mbar_expect_tx(fb, (uint32_t)L::KV_BYTES);
          if (p < n_table) sm100::tma_load_5d(dst, tm, fb, 0, 0, 0, kvh, page, pol);
          else sm100::tma_load_4d(dst, tm_loc, fb, 0, item.loc_lo + (p_begin + p - item.n_cache_pages) * PAGE, 0, kvh, pol);
        }
        __syncwarp();
        if (++s == stages) { s = 0; ph ^= 1u; }
      }
    }
  } else if (warp == 1) {
    // ===================== MMA issuer =====================
    // Runs the same schedule as the watcher to the end whatever happens, one barrier operation each per event.
    const uint32_t idesc_qk = sm100::make_idesc_bf16(128, PAGE);
    const uint32_t idesc_pv = sm100::make_idesc_bf16(128, HD) | (1u << 16);      // B (= V) is MN-major
    // descriptors are built once; the issue loop only adds 16-byte-unit offsets
    const uint64_t q_desc = sm100::make_desc_sw128(smem0 + L::Q_OFF);
    const uint64_t k_desc0 = sm100::make_desc_sw128(smem0 + L::K_OFF);
    const uint64_t v_desc0 = sm100::make_desc_sw128_mn(smem0 + L::V_OFF, PAGE * 128);
    constexpr uint64_t KV16 = L::KV_BYTES >> 4, Q16 = L::Q_BYTES >> 4;
    // scores of page p (ring stage s) for stream t, into S buffer b
    auto issue_qk = [&](int t, int b, int s) {
      const uint64_t qd = q_desc + (pair && t ? Q16 : 0), kd = k_desc0 + (uint64_t)s * KV16;
      const uint32_t d = tmem_S + (uint32_t)((t * 2 + b) * PAGE);
#pragma unroll
      for (int kk = 0; kk < HD / 16; ++kk)             // 64-element half kk / 4 of the head, 16 elements of it
        sm100::mma_bf16_ss(d, qd + (kk / 4) * (128 * 128 / 16) + (kk % 4) * 2, kd + (kk / 4) * (PAGE * 128 / 16) + (kk % 4) * 2, idesc_qk, kk > 0 ? 1u : 0u);
    };
    for (int p = 0; p < min(ahead, np); ++p) {
      sm100::named_bar_sync(9u + (uint32_t)p, 64);
      sm100::tc_fence_after();
      if (sm100::elect_one()) {
        for (int t = stream0(p); t < stream1(p); ++t) {
          const int b = shared ? p : p >> 1;
          issue_qk(t, b, p);
          sm100::mma_commit(sm100::smem_u32(&ctl.s_full[t][b]));
        }
        sm100::mma_commit(sm100::smem_u32(&ctl.k_empty[p]));
      }
      __syncwarp();
    }
    int sv = 0, sk = ahead % L::K_STAGES;              // ring stages of V(p) and K(p + ahead)
    for (int p = 0; p < np; ++p) {
      const int j = shared ? p : p >> 1, b = j & 1;
      const uint64_t vd = v_desc0 + (uint64_t)sv * KV16;
      for (int t = stream0(p); t < stream1(p); ++t) {
        const bool last_stream = !pair || t == 1;
        sm100::named_bar_sync(1u + (uint32_t)(t * 2 + b), 64);
        sm100::tc_fence_after();
        if (sm100::elect_one()) {
          const uint32_t p_tmem = tmem_S + (uint32_t)((t * 2 + b) * PAGE), o_tmem = tmem_O + (uint32_t)(t * HD);
#pragma unroll
          for (int kk = 0; kk < PAGE / 16; ++kk)       // 16 keys per instruction: 8 columns of P, 16 V rows (2048 B)
            sm100::mma_bf16_ts(o_tmem, p_tmem + kk * 8, vd + kk * (16 * 128 / 16), idesc_pv, (j > 0 || kk > 0) ? 1u : 0u);
          if (last_stream) sm100::mma_commit(sm100::smem_u32(&ctl.v_empty[sv]));
          if (p + ahead < np) {
            issue_qk(t, b, sk);
            if (last_stream) sm100::mma_commit(sm100::smem_u32(&ctl.k_empty[sk]));
          }
          sm100::mma_commit(sm100::smem_u32(&ctl.s_full[t][b]));       // step j + 2's scores, or only "P V of step j is done"
        }
        __syncwarp();
      }
      if (++sv == L::V_STAGES) sv = 0;
      if (++sk == L::K_STAGES) sk = 0;
    }
  } else if (warp == 2) {
    // ===================== watcher =====================
    // Waits (bounded) for what each group of MMAs needs and arrives on the group's hardware barrier.  A barrier
    // cannot be arrived on twice before the MMA warp has passed it: P of step j + 2 needs the scores whose products
    // are issued behind step j's.  After a failed wait that argument no longer holds, so from then on the watcher
    // meets the MMA warp at every barrier instead.
    bool failed = false;
    auto release = [&](uint32_t id, uint32_t bar0, uint32_t par0, uint32_t bar1, uint32_t par1, uint32_t bar2, uint32_t par2) {
      if (!failed) {
        bool ok = true;
        if (lane == 0)
          ok = (!bar1 || sm100::mbar_wait(bar1, par1, abortp)) && (!bar2 || sm100::mbar_wait(bar2, par2, abortp)) && sm100::mbar_wait(bar0, par0, abortp);
        failed = !__shfl_sync(0xffffffffu, ok, 0);
      }
      if (!failed) sm100::named_bar_arrive(id, 64);
      else sm100::named_bar_sync(id, 64);
    };
    for (int p = 0; p < min(ahead, np); ++p)
      release(9u + (uint32_t)p, sm100::smem_u32(&ctl.k_full[p]), 0, p ? 0u : sm100::smem_u32(&ctl.q_full), 0, 0u, 0);
    int sv = 0, sk = ahead % L::K_STAGES; uint32_t phv = 0, phk = (uint32_t)(ahead / L::K_STAGES) & 1u;
    for (int p = 0; p < np; ++p) {
      const int j = shared ? p : p >> 1, b = j & 1;
      for (int t = stream0(p); t < stream1(p); ++t) {
        const bool first_stream = !pair || t == 0;
        release(1u + (uint32_t)(t * 2 + b), sm100::smem_u32(&ctl.p_full[t][b]), (uint32_t)(j >> 1) & 1u, first_stream ? sm100::smem_u32(&ctl.v_full[sv]) : 0u, phv,
                first_stream && p + ahead < np ? sm100::smem_u32(&ctl.k_full[sk]) : 0u, phk);
      }
      if (++sv == L::V_STAGES) { sv = 0; phv ^= 1u; }
      if (++sk == L::K_STAGES) { sk = 0; phk ^= 1u; }
    }
  } else if (warp >= 4) {
    // ===================== softmax =====================
    const int tile = pair ? t : 0;
    const int nj = shared ? np : (np + 1 - t) >> 1;      // steps of this stream
    // (a row without a slot sees everything, so that its warp does not mask page after page for it)
    int my_nvis = 0x7fffffff, my_loc0 = item.loc_lo, my_nloc = 1 << 30;
    {
      const int pr = row0 + tile * a.spt + my_row / a.G;
      if (my_row < rows_used && pr < item.row_end) {
        my_slot = pr;
        if constexpr (DIRECT) { const RowKeys w = step_row_keys(a.direct.seq_len, a.direct.k, a.direct.n_max, pr); my_nvis = w.nvis; my_nloc = w.nloc; my_loc0 = w.loc0; }
        else { my_nvis = a.nvis[pr]; my_nloc = a.nloc[pr]; my_loc0 = a.loc0[pr]; }
      }
    }
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t s_addr0 = tmem_S + (uint32_t)(t * 2 * PAGE) + lane_addr, o_addr = tmem_O + (uint32_t)(t * HD) + lane_addr;
    const uint32_t s_bar0 = sm100::smem_u32(&ctl.s_full[t][0]), p_bar0 = sm100::smem_u32(&ctl.p_full[t][0]);
    // wait until the scores of step j are there (for j >= nj: until P V of step j - 2 is done).  A parity wait means what it says
    // because the barrier's next completion needs a P that this warp has not yet written.
    auto wait_s = [&](int j) { return sm100::mbar_wait_warp(s_bar0 + (uint32_t)(j & 1) * 8u, (uint32_t)(j >> 1) & 1u, abortp); };
    float m_ref = -INFINITY, l_run = 0.f;
    bool ok = true;
#pragma unroll 1
    for (int j = AHEAD ? -1 : 0; j < nj; ++j) {          // (step -1: the walk)
      const bool live = !AHEAD || j >= 0;
      if (live) {
        if (!(ok = wait_s(j))) break;
        sm100::tc_fence_after();
      }
      const uint32_t s_addr = s_addr0 + (uint32_t)((j & 1) * PAGE);
      uint32_t sv[2][32];
      sm100::tmem_ld32(s_addr, sv[0]);
      sm100::tmem_ld32(s_addr + 32, sv[1]);
      sm100::tmem_wait_ld();
      // Visible keys of the page for my row: [lo, hi) in page-local indices.  Masking is skipped
      // for pages that are visible in full (all cached pages but the last ones of a row).
      {
        const int p = p_begin + (shared ? j : 2 * j + t);
        int lo = 0, hi = 0;
        if (!live) { }
        else if (p < item.n_cache_pages) hi = my_nvis - p * PAGE;
        else if (my_nloc > 0) { lo = my_loc0 - (item.loc_lo + (p - item.n_cache_pages) * PAGE); hi = lo + my_nloc; }
        if (lo > 0 || hi < PAGE) {
#pragma unroll
          for (int c = 0; c < PAGE; ++c)
            if (c < lo || c >= hi) sv[c / 32][c & 31] = 0xff800000u;               // -inf
        }
      }
      // Softmax in base 2.  The scores stay raw: the scale is applied inside one FMA per two elements (s * scale - m), and
      // the max and the sum run as independent chains.
      float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int c = 0; c < 64; c += 2) mx4[(c >> 1) & 3] = sm100::max3(mx4[(c >> 1) & 3], __uint_as_float(sv[c / 32][c & 31]), __uint_as_float(sv[c / 32][(c & 31) + 1]));
      const float mx = sm100::max3(mx4[0], mx4[1], fmaxf(mx4[2], mx4[3])) * a.scale_log2;      // scale > 0; -inf stays -inf
      // raise the reference only when this step exceeds it by more than the threshold
      // (-inf + threshold = -inf, so the first visible key always sets it)
      const float m_new = (mx > m_ref + RAISE_THRESHOLD) ? mx : m_ref;
      const float alpha = (m_new == m_ref) ? 1.f : exp2f(m_ref - m_new);      // m_ref = -inf gives 0
      const float neg_m = (m_new == -INFINITY) ? 0.f : -m_new;
      m_ref = live ? m_new : m_ref;
      if (j > 0 && __any_sync(0xffffffffu, alpha != 1.f)) {
        // O is rescaled in place: P V of step j - 1 must be done; that of step j waits for P
        if (!(ok = wait_s(j + 1))) break;
        sm100::tc_fence_after();
#pragma unroll 2
        for (int c = 0; c < HD / 16; ++c) {
          uint32_t v[16];
          sm100::tmem_ld16(o_addr + c * 16, v);
          sm100::tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * alpha);
          sm100::tmem_st16(o_addr + c * 16, v);
        }
      }
      const sm100::f32x2 scale2 = sm100::pack2(a.scale_log2, a.scale_log2), neg_m2 = sm100::pack2(neg_m, neg_m);
      sm100::f32x2 sum2[2] = {0ull, 0ull};           // (0, 0)
      uint32_t pk[32];
#pragma unroll
      for (int c = 0; c < 64; c += 2) {
        float x, y;
        sm100::unpack2(sm100::fma2(sm100::pack2(__uint_as_float(sv[c / 32][c & 31]), __uint_as_float(sv[c / 32][(c & 31) + 1])), scale2, neg_m2), x, y);
        x = sm100::ex2_approx(x); y = sm100::ex2_approx(y);           // -inf -> 0
        sum2[(c >> 1) & 1] = sm100::add2(sum2[(c >> 1) & 1], sm100::pack2(x, y));
        __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
        pk[c >> 1] = *reinterpret_cast<uint32_t *>(&h);
      }
      if (live) {
        sm100::tmem_st32(s_addr, pk);
        sm100::tmem_wait_st();
        sm100::tc_fence_before();
        __syncwarp();
        if (lane == 0) sm100::mbar_arrive(p_bar0 + (uint32_t)(j & 1) * 8u);
      }
      float sa, sb;
      sm100::unpack2(sm100::add2(sum2[0], sum2[1]), sa, sb);
      l_run = live ? l_run * alpha + (sa + sb) : 0.f;
    }
    // ---- output: O is complete once the last P V has finished ----
    if constexpr (CLUSTER) sm100::cluster_wait();        // the cluster's other CTAs run
    pdl_wait();                                          // (long over; the stores below must not overtake it formally either)
    if (ok && nj > 1) ok = wait_s(nj);                   // (P V of the last step but one; in order, so that the parity wait below is unambiguous)
    if (ok && nj > 0) ok = wait_s(nj + 1);
    sm100::tc_fence_after();
    bf16 *o = a.O + ((size_t)max(my_slot, 0) * a.Hq + kvh * a.G + my_row % a.G) * HD;
    const size_t part = (size_t)blockIdx.x * 2 + tile;
    float *po = a.part_O + (part * (HD / 4) * 128 + my_row) * 4;
    auto write32 = [&](const float (&v)[32], int col, float inv) {       // columns [col, col + 32) of this row
      if (my_slot < 0) return;
      if (!item.split) {
#pragma unroll
        for (int i = 0; i < 32; i += 8) {
          uint4 u;
          __nv_bfloat162 h0 = __floats2bfloat162_rn(v[i] * inv, v[i + 1] * inv), h1 = __floats2bfloat162_rn(v[i + 2] * inv, v[i + 3] * inv),
                         h2 = __floats2bfloat162_rn(v[i + 4] * inv, v[i + 5] * inv), h3 = __floats2bfloat162_rn(v[i + 6] * inv, v[i + 7] * inv);
          u.x = *reinterpret_cast<uint32_t *>(&h0); u.y = *reinterpret_cast<uint32_t *>(&h1);
          u.z = *reinterpret_cast<uint32_t *>(&h2); u.w = *reinterpret_cast<uint32_t *>(&h3);
          *reinterpret_cast<uint4 *>(o + col + i) = u;
        }
      } else {
#pragma unroll
        for (int i = 0; i < 32; i += 4)
          *reinterpret_cast<float4 *>(po + (size_t)((col + i) / 4) * (128 * 4)) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
      }
    };
    auto load32 = [&](int col, float (&v)[32]) {
      uint32_t w[32];
      sm100::tmem_ld32(o_addr + col, w);
      sm100::tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(w[i]);
    };
    if (shared) {
      if (ok && nj > 0) {
        const float inv = item.split ? 1.f : 1.f / l_run;
#pragma unroll
        for (int c = 0; c < HD; c += 32) { float v[32]; load32(c, v); write32(v, c, inv); }
        if (my_slot >= 0 && item.split) a.part_ml[part * 128 + my_row] = make_float2(m_ref, l_run);
      }
    } else if (CLUSTER && sharing ? np_item > 0 : np > 0) {
      // The streams' halves of the same rows: each hands the other's columns over and finishes its own.  All MMAs have
      // read the K/V rings once every warp has got here (a failed stream only has to show up).
      float4 *xo = reinterpret_cast<float4 *>(smem_raw + L::XCHG_OFF);   // [stream that reads][HD / 8][128]
      float2 *xml = reinterpret_cast<float2 *>(smem_raw + L::XCHG_ML_OFF);
      sm100::named_bar_sync(13, 256);
      if (ok) {
        xml[t * 128 + my_row] = make_float2(m_ref, l_run);
#pragma unroll
        for (int c = 0; c < HD / 2; c += 32) {
          float v[32];
          if (nj > 0) load32((1 - t) * (HD / 2) + c, v);
          else {
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = 0.f;
          }
#pragma unroll
          for (int i = 0; i < 32; i += 4) xo[((1 - t) * (HD / 8) + (c + i) / 4) * 128 + my_row] = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        }
      }
      sm100::named_bar_sync(13, 256);
      if (ok && (!CLUSTER || sharing)) {
        const float2 other = xml[(1 - t) * 128 + my_row];
        const float M = fmaxf(m_ref, other.x);
        const float wm = m_ref == -INFINITY ? 0.f : exp2f(m_ref - M), wo = other.x == -INFINITY ? 0.f : exp2f(other.x - M);
        const float l = wm * l_run + wo * other.y, inv = CLUSTER || item.split ? 1.f : 1.f / l;
#pragma unroll
        for (int c = 0; c < HD / 2; c += 32) {
          float v[32];
          if (nj > 0) load32(t * (HD / 2) + c, v);
          else {
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = 0.f;
          }
#pragma unroll
          for (int i = 0; i < 32; i += 4) {
            const float4 x = xo[(t * (HD / 8) + (c + i) / 4) * 128 + my_row];
            v[i] = wm * v[i] + wo * x.x; v[i + 1] = wm * v[i + 1] + wo * x.y; v[i + 2] = wm * v[i + 2] + wo * x.z; v[i + 3] = wm * v[i + 3] + wo * x.w;
          }
          if constexpr (CLUSTER) {
            if (my_slot >= 0) {
#pragma unroll
              for (int i = 0; i < 32; i += 4) {
                const int owner = (c + i) >> c_shift, at = (c + i) & (c_cols - 1);
                sm100::st_cluster_v4(sm100::cluster_addr(smem0 + L::PEER_OFF, (uint32_t)owner) + (uint32_t)((((c_rank * 2 + t) * (c_cols / 4) + at / 4) * 128 + my_row) * 16),
                                     v[i], v[i + 1], v[i + 2], v[i + 3]);
              }
            }
          } else {
            write32(v, t * (HD / 2) + c, inv);
          }
        }
        if constexpr (CLUSTER) {
          if (t == 0 && my_slot >= 0)
            for (int r = 0; r < c_size; ++r) sm100::st_cluster_v2(sm100::cluster_addr(smem0 + L::PEER_ML_OFF, (uint32_t)r) + (uint32_t)((c_rank * 128 + my_row) * 8), M, l);
        } else {
          if (t == 0 && my_slot >= 0 && item.split) a.part_ml[part * 128 + my_row] = make_float2(M, l);
        }
      }
      if constexpr (CLUSTER && DIRECT) {
        if (ok && !sharing) finish_alone<HD>(o_addr, t, my_row, m_ref, l_run, nj, my_slot < 0 ? nullptr : o, xo, xml);
      }
    }
  }
  if constexpr (CLUSTER) {
    if (warp < 4) sm100::cluster_wait();
    if (sharing) sm100::cluster_sync();                  // the stores to one another have arrived
    if (sharing && warp >= 4 && np_item > 0 && my_slot >= 0) {
      const float2 *ml = reinterpret_cast<const float2 *>(smem_raw + L::PEER_ML_OFF) + my_row;
      const float4 *x = reinterpret_cast<const float4 *>(smem_raw + L::PEER_OFF) + t * (c_cols / 4) * 128 + my_row;
      float M = -INFINITY, den = 0.f;
      for (int r = 0; r < c_size; ++r) M = fmaxf(M, ml[r * 128].x);
      for (int r = 0; r < c_size; ++r) den += exp2f(ml[r * 128].x - M) * ml[r * 128].y;
      const float inv = 1.f / den;
      bf16 *o = a.O + ((size_t)my_slot * a.Hq + kvh * a.G + my_row % a.G) * HD + t * (HD / 2) + c_rank * c_cols;
      for (int g = 0; g < c_cols / 4; g += 2) {          // eight columns
        float acc[8] = {};
        for (int r = 0; r < c_size; ++r) {
          const float w = exp2f(ml[r * 128].x - M);      // (a CTA without pages: 0)
          const float4 u = x[(r * 2 * (c_cols / 4) + g) * 128], v = x[(r * 2 * (c_cols / 4) + g + 1) * 128];
          acc[0] = fmaf(w, u.x, acc[0]); acc[1] = fmaf(w, u.y, acc[1]); acc[2] = fmaf(w, u.z, acc[2]); acc[3] = fmaf(w, u.w, acc[3]);
          acc[4] = fmaf(w, v.x, acc[4]); acc[5] = fmaf(w, v.y, acc[5]); acc[6] = fmaf(w, v.z, acc[6]); acc[7] = fmaf(w, v.w, acc[7]);
        }
        __nv_bfloat162 h0 = __floats2bfloat162_rn(acc[0] * inv, acc[1] * inv), h1 = __floats2bfloat162_rn(acc[2] * inv, acc[3] * inv),
                       h2 = __floats2bfloat162_rn(acc[4] * inv, acc[5] * inv), h3 = __floats2bfloat162_rn(acc[6] * inv, acc[7] * inv);
        uint4 w4;
        w4.x = *reinterpret_cast<uint32_t *>(&h0); w4.y = *reinterpret_cast<uint32_t *>(&h1);
        w4.z = *reinterpret_cast<uint32_t *>(&h2); w4.w = *reinterpret_cast<uint32_t *>(&h3);
        *reinterpret_cast<uint4 *>(o + g * 4) = w4;
      }
    }
  }

  // ---- teardown ----
  sm100::tc_fence_before();
  __syncthreads();
  if (ctl.abort_flag) {
    if (threadIdx.x == 0 && a.status) atomicExch(a.status, 2);
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == 1) {
    __syncwarp();
    sm100::tc_fence_after();
    sm100::tmem_dealloc(tmem, L::TMEM_COLS);
  }
  if (threadIdx.x == 0) tl_end(tl);
}

// Merge the partial results of the query tiles that were split: O = sum_s 2^(m_s - M) O_s / sum_s 2^(m_s - M) l_s.
// HD / 16 blocks of 256 threads per (query tile, KV head); a thread takes 8 columns of one MMA row, neighbouring
// threads neighbouring rows, which is how the partial results lie in memory.
template <int HD, bool DIRECT>
__global__ void __launch_bounds__(256)
attn_combine_kernel(const Args a, TlSlot tl) {
  pdl_trigger();
  if (DIRECT || !a.early) pdl_wait();
  constexpr int BLOCKS = HD / 16;
  const int w = blockIdx.x / BLOCKS, kvh = w % a.Hkv;
  const int cg = (blockIdx.x % BLOCKS) * 2 + (threadIdx.x >> 7), m = threadIdx.x & 127;
  Tile t{};
  if constexpr (DIRECT) {
    const Item it = direct_tile(a, w / a.Hkv);
    t.row0 = it.row0; t.row_end = it.row_end; t.n_items = direct_pieces(a, it.p_end); t.item0 = w / a.Hkv * a.direct.pieces;
  } else {
    t = a.tiles[w / a.Hkv];
  }
  const int slot = t.row0 + m / a.G;
  pdl_wait();
  if (threadIdx.x == 0) tl_go(tl);
  if (t.n_items > 1 && m < a.spt * a.G && slot < t.row_end) {
    const size_t part = ((size_t)t.item0 * a.Hkv + kvh) * 2 + t.sub;
    const float2 *ml = a.part_ml + part * 128 + m;
    const float4 *po = reinterpret_cast<const float4 *>(a.part_O) + part * (HD / 4) * 128 + (size_t)cg * 2 * 128 + m;
    const size_t ml_step = (size_t)a.Hkv * 2 * 128, po_step = (size_t)a.Hkv * 2 * (HD / 4) * 128;
    // four partial results at a time, all their loads before the first use; the running sum is rescaled when the maximum rises
    float M = -INFINITY, den = 0.f;
    float acc[8] = {};
    for (int s0 = 0; s0 < t.n_items; s0 += 4) {
      float2 v[4]; float4 x[4], y[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        v[u] = make_float2(-INFINITY, 0.f);
        x[u] = y[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s0 + u < t.n_items) { v[u] = ml[(s0 + u) * ml_step]; x[u] = po[(s0 + u) * po_step]; y[u] = po[(s0 + u) * po_step + 128]; }
      }
      const float M_new = fmaxf(fmaxf(M, fmaxf(v[0].x, v[1].x)), fmaxf(v[2].x, v[3].x));
      const float keep = M == -INFINITY ? 0.f : exp2f(M - M_new);
      M = M_new;
      den *= keep;
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[j] *= keep;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float wgt = v[u].x == -INFINITY ? 0.f : exp2f(v[u].x - M);
        den += wgt * v[u].y;
        acc[0] = fmaf(wgt, x[u].x, acc[0]); acc[1] = fmaf(wgt, x[u].y, acc[1]); acc[2] = fmaf(wgt, x[u].z, acc[2]); acc[3] = fmaf(wgt, x[u].w, acc[3]);
        acc[4] = fmaf(wgt, y[u].x, acc[4]); acc[5] = fmaf(wgt, y[u].y, acc[5]); acc[6] = fmaf(wgt, y[u].z, acc[6]); acc[7] = fmaf(wgt, y[u].w, acc[7]);
      }
    }
    const float inv = 1.f / den;
    __nv_bfloat162 h0 = __floats2bfloat162_rn(acc[0] * inv, acc[1] * inv), h1 = __floats2bfloat162_rn(acc[2] * inv, acc[3] * inv),
                   h2 = __floats2bfloat162_rn(acc[4] * inv, acc[5] * inv), h3 = __floats2bfloat162_rn(acc[6] * inv, acc[7] * inv);
    uint4 u;
    u.x = *reinterpret_cast<uint32_t *>(&h0); u.y = *reinterpret_cast<uint32_t *>(&h1);
    u.z = *reinterpret_cast<uint32_t *>(&h2); u.w = *reinterpret_cast<uint32_t *>(&h3);
    *reinterpret_cast<uint4 *>(a.O + ((size_t)slot * a.Hq + kvh * a.G + m % a.G) * HD + cg * 8) = u;
  }
  if (threadIdx.x == 0) tl_end(tl);
}

}  // namespace attn_tc
