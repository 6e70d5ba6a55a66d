// Slot assembly, embedding, RMSNorm, RoPE + KV placement, SwiGLU, argmax,
// draft/verify and KV commit kernels of the TiDAR decode step.
#pragma once
#include "common.cuh"
#include "sm100_ptx.cuh"
#include "attn_tc.cuh"

// Four consecutive split-K partial sums starting at p (fp32 or bf16 slabs).
template <typename T> __device__ __forceinline__ float4 load4(const T *p);
template <> __device__ __forceinline__ float4 load4<float>(const float *p) { return *reinterpret_cast<const float4 *>(p); }
template <> __device__ __forceinline__ float4 load4<bf16>(const bf16 *p) {
  const uint2 u = *reinterpret_cast<const uint2 *>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}

// v += the S (at most MAX_SLABS) partial sums at p, p + stride, ..., in that order.  AT_ONCE loads are issued before their
// first addition: with one load per turn of a loop over S, the kernels that read slabs spent most of their time waiting
// (norm 3.6 -> 2.0 us at 272 rows of 1536).
constexpr int MAX_SLABS = 8;
template <int AT_ONCE, int MOST = MAX_SLABS, typename SLAB>
__device__ __forceinline__ void add_slabs(float4 &v, const SLAB *__restrict__ p, int S, size_t stride) {
#pragma unroll
  for (int s0 = 0; s0 < MOST; s0 += AT_ONCE) {
    if (s0 >= S) break;
    float4 q[AT_ONCE];
#pragma unroll
    for (int u = 0; u < AT_ONCE; ++u)
      if (s0 + u < S) q[u] = load4<SLAB>(p + (s0 + u) * stride);
#pragma unroll
    for (int u = 0; u < AT_ONCE; ++u)
      if (s0 + u < S) { v.x += q[u].x; v.y += q[u].y; v.z += q[u].z; v.w += q[u].w; }
  }
}

// One embedding row (bf16, d a multiple of 8) -> fp32, 16-byte loads.
__device__ __forceinline__ void embed_row_to_f32(const bf16 *__restrict__ e, float *__restrict__ x, int d) {
  for (int c = threadIdx.x * 8; c < d; c += blockDim.x * 8) {
    const uint4 u = *reinterpret_cast<const uint4 *>(e + c);
    const __nv_bfloat162 *p = reinterpret_cast<const __nv_bfloat162 *>(&u);
    const float2 a = __bfloat1622float2(p[0]), b = __bfloat1622float2(p[1]), cc = __bfloat1622float2(p[2]), dd = __bfloat1622float2(p[3]);
    *reinterpret_cast<float4 *>(x + c) = make_float4(a.x, a.y, b.x, b.y);
    *reinterpret_cast<float4 *>(x + c + 4) = make_float4(cc.x, cc.y, dd.x, dd.y);
  }
}

// ---------------------------------------------------------------------------
// Slot assembly + embedding gather for a decode step.
// Slot layout per sequence (k causal slots, then n_blocks blocks of k mask slots;
// paper Section 3.3 footnote, figure "TiDAR Attention Masks"):
//   causal j       : token block[j], position n+j
//   mask (b, i)    : [MASK], position n+b+1+i (no label shift: a mask slot predicts
//                    its own position; paper Section 4.4.3)
// n_blocks = k for a TiDAR step; n_blocks = 0 for a plain autoregressive step (the
// causal section alone: paper Section 3.1, the model keeps its autoregressive mode).
// The step may use a block length k that differs from the one the previous pass left
// (blk_len[seq] valid entries): drafts the sequence does not have are fed as [MASK]
// and can never be accepted (see verify_select_kernel).
// The listed sequences may use different block lengths in one step: step_k[s] is sequence s's,
// step_off[s] its first row and step_loc[s] its first step-local K/V row (null: all use k).
// One block per row; also snapshots n into step_n for the commit kernel.
// ---------------------------------------------------------------------------
struct StepLayout { const int32_t *k, *off, *loc; int n_seqs; };     // per listed sequence; k == null: uniform

// A step's exchange with the host goes through pinned host memory that the kernels read and write themselves: two slots,
// used in turn (a second step may be enqueued while the first runs).  turn: device word, the number of steps run.
// (Four small copies around the kernels cost a one-sequence step of the tiny model 40 of its 160 us.)
struct StepIo {
  int32_t *turn, *blocks_done, *status;                      // device
  const int32_t *in[2];                                      // [2][max_batch]: listed sequences, forced lengths
  int32_t *out[2];                                           // [n_seqs][k_max + 1]: L, tokens
  int32_t *done[2];                                          // [0] = turn + 1 (the step ran to its end), [1] = status
  int32_t max_batch;
};

// The step's inputs to device memory, and for a step of mixed block lengths its layout (n_head > 0): h_lay holds n_head ints and
// two tables of cap entries, n_units of them in use, in the same order as the device arrays at lay.  One block.
__global__ void __launch_bounds__(256) stage_step_kernel(StepIo io, int n_seqs, int32_t *__restrict__ step_seqs, int32_t *__restrict__ forced,
                                                         const int32_t *__restrict__ h_lay, int32_t *__restrict__ lay, int n_head, int cap, int n_units, TlSlot tl) {
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0) tl_go(tl);
  const int32_t *in = io.in[*io.turn & 1];
  for (int i = threadIdx.x; i < n_seqs; i += blockDim.x) {
    const int a = in[i], b = in[io.max_batch + i];
    step_seqs[i] = a; forced[i] = b;
  }
  if (n_head > 0)
    for (int i = threadIdx.x; i < n_head + 2 * n_units; i += blockDim.x) {
      const int j = i - n_head, at = j < n_units ? i : i + cap - n_units;
      lay[at] = h_lay[at];
    }
  if (threadIdx.x == 0) tl_end(tl);
}

__global__ void assemble_step_kernel(RowMeta m, const int32_t *__restrict__ step_seqs, const int32_t *__restrict__ seq_len,
                                     const int32_t *__restrict__ block_ids, const int32_t *__restrict__ blk_len, int k, int n_blocks,
                                     StepLayout lay, int k_max, int mask_id,
                                     int32_t *__restrict__ step_n, const bf16 *__restrict__ embed, int d,
                                     float *__restrict__ X, int sampling, unsigned long long seed, TlSlot tl) {
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0) tl_go(tl);
  const int r = blockIdx.x;
  int s, slot, loc_base;
  if (lay.k && r >= lay.off[lay.n_seqs]) {       // a row that only fills the last 16 rows up: no sequence, no K/V, seen by nothing
    if (threadIdx.x == 0) {
      m.seq[r] = 0; m.ids[r] = mask_id; m.pos[r] = 0; m.nvis[r] = 0; m.loc0[r] = 0; m.nloc[r] = 0; m.cache_pos[r] = -1; m.local_idx[r] = -1;
      if (sampling) m.skey[r] = 0;
      tl_end(tl);
    }
    for (int c = threadIdx.x; c < d; c += blockDim.x) X[(size_t)r * d + c] = 0.f;
    return;
  }
  if (lay.k) {                                   // per-sequence block lengths: find the sequence this row belongs to
    s = 0;
    while (s + 1 < lay.n_seqs && r >= lay.off[s + 1]) ++s;
    k = lay.k[s]; n_blocks = k; slot = r - lay.off[s]; loc_base = lay.loc[s];
  } else {
    const int T = k * (n_blocks + 1);
    s = r / T; slot = r % T; loc_base = s * k * k;
  }
  const int seq = step_seqs[s];
  const int n = seq_len[seq];
  int id;
  if (slot < k && slot < blk_len[seq]) id = block_ids[seq * k_max + slot]; else id = mask_id;
  if (threadIdx.x == 0) {
    if (slot == 0) step_n[s] = n;
    m.seq[r] = seq;
    m.ids[r] = id;
    if (slot < k) {
      m.pos[r] = n + slot; m.nvis[r] = n + slot + 1; m.loc0[r] = 0; m.nloc[r] = 0;
      m.cache_pos[r] = n + slot; m.local_idx[r] = -1;
      if (sampling) m.skey[r] = position_key(seed, seq, n + slot + 1);        // a causal slot predicts the next position
    } else {
      const int b = (slot - k) / k, i = (slot - k) % k;
      m.pos[r] = n + b + 1 + i; m.nvis[r] = n + b + 1; m.loc0[r] = loc_base + b * k; m.nloc[r] = k;
      m.cache_pos[r] = -1; m.local_idx[r] = loc_base + b * k + i;
      if (sampling) m.skey[r] = position_key(seed, seq, n + b + 1 + i);       // a mask slot predicts its own position
    }
  }
  embed_row_to_f32(embed + (size_t)id * d, X + (size_t)r * d, d);
  if (threadIdx.x == 0) tl_end(tl);
}

// Prefill chunk: rows g = row0 .. row0+rows-1 of [prompt ; k mask tokens]
// (paper Section 3.2, Appendix B): prompt rows causal, mask rows see the whole
// prompt and each other.
__global__ void assemble_prefill_kernel(RowMeta m, int seq, int row0, int n_prompt, int k, int mask_id,
                                        const int32_t *__restrict__ prompt, const bf16 *__restrict__ embed, int d,
                                        float *__restrict__ X, int sampling, unsigned long long seed) {
  const int r = blockIdx.x;
  const int g = row0 + r;
  const int id = g < n_prompt ? prompt[g] : mask_id;
  if (threadIdx.x == 0) {
    m.seq[r] = seq; m.ids[r] = id; m.pos[r] = g;
    if (g < n_prompt) {
      m.nvis[r] = g + 1; m.loc0[r] = 0; m.nloc[r] = 0; m.cache_pos[r] = g; m.local_idx[r] = -1;
      if (sampling) m.skey[r] = position_key(seed, seq, g + 1);
    } else {
      m.nvis[r] = n_prompt; m.loc0[r] = 0; m.nloc[r] = k; m.cache_pos[r] = -1; m.local_idx[r] = g - n_prompt;
      if (sampling) m.skey[r] = position_key(seed, seq, g);
    }
  }
  embed_row_to_f32(embed + (size_t)id * d, X + (size_t)r * d, d);
}

// Row metadata of the stand-alone attention entry points.
__global__ void attn_meta_kernel(RowMeta m, const int32_t *__restrict__ seq_len, int k, int R, int n_max) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= R) return;
  const attn_tc::RowKeys w = attn_tc::step_row_keys(seq_len, k, n_max, r);
  m.seq[r] = w.seq; m.nvis[r] = w.nvis; m.loc0[r] = w.loc0; m.nloc[r] = w.nloc;
}
// The same for the tensor-core attention kernel, with its work plan (the first block).
__global__ void __launch_bounds__(512) attn_meta_plan_kernel(RowMeta m, const int32_t *__restrict__ seq_len, int k, int R, int n_max, attn_tc::PlanArgs plan) {
  pdl_trigger();
  pdl_wait();
  if (blockIdx.x == 0) { attn_tc::plan_block(plan, [&](int r) { return attn_tc::step_row_keys(seq_len, k, n_max, r); }); return; }
  const int r = (blockIdx.x - 1) * blockDim.x + threadIdx.x;
  if (r >= R) return;
  const attn_tc::RowKeys w = attn_tc::step_row_keys(seq_len, k, n_max, r);
  m.seq[r] = w.seq; m.nvis[r] = w.nvis; m.loc0[r] = w.loc0; m.nloc[r] = w.nloc;
}

// What every layer of a pass shares, computed once per pass from the row metadata: cos/sin of
// pos * theta^(-2i/hd) (evaluated in double, stored as float), one thread per (row, i), and, when
// plan.tiles is set, the attention work plan (the first block).
__global__ void __launch_bounds__(256) pass_setup_kernel(RowMeta m, int R, int half, double theta,
                                  float *__restrict__ cs, float *__restrict__ sn, attn_tc::PlanArgs plan, TlSlot tl) {
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0) tl_go(tl);
  const int first = plan.tiles ? 1 : 0;
  if (first && blockIdx.x == 0) attn_tc::plan_block(plan, [&](int r) { return attn_tc::RowKeys{m.nvis[r], m.loc0[r], m.nloc[r], m.seq[r]}; });
  else {
    const int t = (blockIdx.x - first) * blockDim.x + threadIdx.x;
    if (t < R * half) {
      const int r = t / half, i = t % half;
      const double inv = pow(theta, -(double)i / (double)half);
      double s, c;
      sincos((double)m.pos[r] * inv, &s, &c);
      cs[t] = (float)c; sn[t] = (float)s;
    }
  }
  if (threadIdx.x == 0) tl_end(tl);
}

// ---------------------------------------------------------------------------
// Residual update + RMSNorm.  X (fp32 residual stream) += sum over the S split-K
// partial results of the previous projection (fixed order: deterministic), then
// A = bf16(X * rsqrt(mean(X^2) + eps) * gain).  One block per row; a thread keeps NV
// groups of four columns in registers (NV * 4 * THREADS >= d).
// ---------------------------------------------------------------------------
// SLABS: the most partial results there can be (1 or MAX_SLABS: with one, four blocks of a many-row pass fit on an SM).
// WALK (passes of few rows, whose blocks are resident long before their input is ready): the block goes through everything twice, the first time
// ahead of the wait, with the loads from its output buffer, which it reads nowhere else, and nothing stored.  That brings the code into the
// instruction cache, from which a layer's other kernels push it between two launches.  (8 rows of 1536: 1.5 - 1.8 us behind a gap of 1.35 -> 1.3 - 1.4
// behind 0.8; 20 rows of 4096: gap 1.35 -> 0.85.  With many rows the blocks start late and the walk is in their way: 272 rows of 1536 1.8 -> 3.0 us.)
template <int THREADS, int NV, int SLABS, bool WALK, typename SLAB>
__global__ void __launch_bounds__(THREADS, SLABS == 1 && NV <= 2 && !WALK ? 4 : 1)
rmsnorm_reduce_kernel(float *__restrict__ X, const SLAB *__restrict__ partials, int S, size_t partial_stride,
                      const bf16 *__restrict__ gain, float eps, int d, bf16 *A, TlSlot tl) {
  pdl_trigger();
  __shared__ float red[THREADS / 32];
  const int r = blockIdx.x;
  uint2 gb[NV];                                  // weights: no need to wait for the previous kernel
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int c = (i * THREADS + threadIdx.x) * 4;
    gb[i] = c < d ? *reinterpret_cast<const uint2 *>(gain + c) : make_uint2(0u, 0u);
  }
  float *xr = X + (size_t)r * d;
#pragma unroll 1
  for (int walk = WALK ? 0 : 1; walk < 2; ++walk) {
    const bool live = !WALK || walk != 0;
    if (live) {
      pdl_wait();
      if (threadIdx.x == 0) tl_go(tl);
    }
    const float *x = live ? xr : reinterpret_cast<const float *>(A);
    const SLAB *p = live ? partials + (size_t)r * d : reinterpret_cast<const SLAB *>(A);
    const size_t stride = live ? partial_stride : 0;
    float4 v[NV];
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = (i * THREADS + threadIdx.x) * 4, at = live ? c : 0;
      v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (c < d) {
        v[i] = *reinterpret_cast<const float4 *>(x + at);
        add_slabs<SLABS, SLABS>(v[i], p + at, S, stride);
      }
      ss += v[i].x * v[i].x + v[i].y * v[i].y + v[i].z * v[i].z + v[i].w * v[i].w;
    }
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int i = 0; i < THREADS / 32; ++i) tot += red[i];
    const float inv = rsqrtf(tot / (float)d + eps);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = (i * THREADS + threadIdx.x) * 4;
      if (c < d) {
        if (live && S > 0) *reinterpret_cast<float4 *>(xr + c) = v[i];
        const float2 g0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&gb[i].x)), g1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&gb[i].y));
        __nv_bfloat162 o0 = __floats2bfloat162_rn(v[i].x * inv * g0.x, v[i].y * inv * g0.y), o1 = __floats2bfloat162_rn(v[i].z * inv * g1.x, v[i].w * inv * g1.y);
        uint2 ob; ob.x = *reinterpret_cast<uint32_t *>(&o0); ob.y = *reinterpret_cast<uint32_t *>(&o1);
        if (live) *reinterpret_cast<uint2 *>(A + (size_t)r * d + c) = ob;
      }
    }
    if (WALK && !live) __syncthreads();            // red is written again
  }
  if (threadIdx.x == 0) tl_end(tl);
}

// The same with the row and its fp32 partial results brought to shared memory by bulk copies, one per source, and added in the same order.  For rows of
// many bytes on every SM (see launch_norm_as), where the loads into registers are bound by how many of them an SM keeps in flight: 272
// rows of 4096 with four slabs, 82 KB each, two per SM, 5.2 - 5.4 us -> 3.8.  Dynamic shared memory: (S + 1) * d floats at least.
template <int THREADS, int NV>
__global__ void __launch_bounds__(THREADS, NV <= 2 ? 2048 / THREADS : 1)
rmsnorm_bulk_kernel(float *__restrict__ X, const float *__restrict__ partials, int S, size_t partial_stride,
                    const bf16 *__restrict__ gain, float eps, int d, bf16 *__restrict__ A, int *status, TlSlot tl) {
  pdl_trigger();
  extern __shared__ __align__(128) uint8_t norm_smem[];
  __shared__ __align__(8) uint64_t full[MAX_SLABS + 1];
  __shared__ float red[THREADS / 32];
  __shared__ int abort_flag;
  const int r = blockIdx.x;
  const float *buf = reinterpret_cast<const float *>(norm_smem);
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s <= S; ++s) sm100::mbar_init(sm100::smem_u32(&full[s]), 1);
    sm100::fence_mbar_init();
  }
  uint2 gb[NV];                                  // weights: no need to wait for the previous kernel
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int c = (i * THREADS + threadIdx.x) * 4;
    gb[i] = c < d ? *reinterpret_cast<const uint2 *>(gain + c) : make_uint2(0u, 0u);
  }
  __syncthreads();
  pdl_wait();
  float *xr = X + (size_t)r * d;
  if (threadIdx.x == 0) {
    tl_go(tl);
    const uint32_t bytes = (uint32_t)d * 4u;
    for (int s = 0; s <= S; ++s) {
      const uint32_t bar = sm100::smem_u32(&full[s]);
      sm100::mbar_expect_tx(bar, bytes);
      sm100::bulk_load(sm100::smem_u32(norm_smem) + (uint32_t)s * bytes, s == 0 ? xr : partials + (size_t)(s - 1) * partial_stride + (size_t)r * d, bytes, bar);
    }
  }
  float4 v[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  bool ok = true;
#pragma unroll 1
  for (int s = 0; s <= S && ok; ++s) {
    ok = sm100::mbar_wait(sm100::smem_u32(&full[s]), 0u, &abort_flag);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = (i * THREADS + threadIdx.x) * 4;
      if (ok && c < d) {
        const float4 q = *reinterpret_cast<const float4 *>(buf + (size_t)s * d + c);
        v[i].x += q.x; v[i].y += q.y; v[i].z += q.z; v[i].w += q.w;
      }
    }
  }
  float ss = 0.f;
#pragma unroll
  for (int i = 0; i < NV; ++i) ss += v[i].x * v[i].x + v[i].y * v[i].y + v[i].z * v[i].z + v[i].w * v[i].w;
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int i = 0; i < THREADS / 32; ++i) tot += red[i];
  const float inv = rsqrtf(tot / (float)d + eps);
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int c = (i * THREADS + threadIdx.x) * 4;
    if (c < d) {
      if (S > 0) *reinterpret_cast<float4 *>(xr + c) = v[i];
      const float2 g0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&gb[i].x)), g1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&gb[i].y));
      __nv_bfloat162 o0 = __floats2bfloat162_rn(v[i].x * inv * g0.x, v[i].y * inv * g0.y), o1 = __floats2bfloat162_rn(v[i].z * inv * g1.x, v[i].w * inv * g1.y);
      uint2 ob; ob.x = *reinterpret_cast<uint32_t *>(&o0); ob.y = *reinterpret_cast<uint32_t *>(&o1);
      *reinterpret_cast<uint2 *>(A + (size_t)r * d + c) = ob;
    }
  }
  if (threadIdx.x == 0) {
    if (abort_flag && status) atomicExch(status, 4);
    tl_end(tl);
  }
  if (abort_flag) {                              // (a copy may still be on its way: the block stays until it has had time to land)
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
  }
}

// ---------------------------------------------------------------------------
// RoPE + KV placement.  Input: S split-K partials of the QKV projection, fp32
// [S][R][(Hq+2Hkv)*hd].  Q heads are rotated and stored bf16 [R][Hq][hd]; K heads are
// rotated, V heads copied; both go to the paged cache at the row's cache position
// (causal slots: kept if accepted, evicted otherwise; paper Section 3.3) or to the
// step-local scratch (mask slots, never cached).  Grid (rows, unit chunks of 256).
// Optional, for checkpoints of the decoder families the paper starts from (Section 4.1):
// bias [(Hq+2Hkv)*hd] added to the projection; qn / kn [hd]: RMSNorm over each Q / K head's
// dimensions before the rotation (the hd/8 threads of a head reduce with shuffles).
// ---------------------------------------------------------------------------
// SLABS: the most partial results there can be (1 or MAX_SLABS: with one, and few registers, a pass of many rows keeps
// three times as many loads in flight).
// WALK (few rows, not in the first layer): everything the layers before this one have used too, row metadata, page table, cos/sin, and the weights,
// is read ahead of the wait, and the code behind the wait is walked through once there, as in the norm, with the partial results' loads from
// the cos/sin table and nothing stored.
template <int SLABS, bool WALK, typename SLAB>
__global__ void __launch_bounds__(256, SLABS == 1 ? 6 : 3)
rope_kv_kernel(const SLAB *__restrict__ partials, int S, size_t partial_stride, int Hq, int Hkv, int hd,
               RowMeta m, const float *__restrict__ cs, const float *__restrict__ sn, KvGeom g,
               bf16 *__restrict__ Q, bf16 *__restrict__ Kpool, bf16 *__restrict__ Vpool,
               bf16 *__restrict__ Kloc, bf16 *__restrict__ Vloc,
               const bf16 *__restrict__ bias, const bf16 *__restrict__ qn, const bf16 *__restrict__ kn, float eps, int let_in, TlSlot tl) {
  // let_in (not in a pass's first layer): the attention kernel may start at once.  Otherwise it is let in behind the wait, as the first layer's must
  // be: it and everything after it then know that what was prepared for the whole pass is there (see attn_tc::Args::early).
  if (let_in) pdl_trigger();
  if (!WALK) {
    pdl_wait();
    if (!let_in) pdl_trigger();
    if (threadIdx.x == 0) tl_go(tl);
  }
  // a work unit is 4 consecutive dims i..i+3 of the first half of one
  // head together with their rotation partners i+hd/2..
  const int r = blockIdx.x, half = hd / 2, upr = half / 4;          // units per head
  const int H = Hq + 2 * Hkv, N = H * hd;
  const int cp = m.cache_pos[r], seq = m.seq[r], li = m.local_idx[r];
  // grid (rows, ceil(units / 256)): one unit per thread, so a row's latency is one round of loads
  const int u = blockIdx.y * blockDim.x + threadIdx.x;
  const bool mine = u < H * upr;
  const int h = mine ? u / upr : 0, i = (u % upr) * 4;
  const bf16 *hn = h < Hq ? qn : (h < Hq + Hkv ? kn : nullptr);
  bf16 *dst = nullptr;                           // (null: a row whose K and V go nowhere)
  const bool rotate = h < Hq + Hkv;
  if (h < Hq) {
    dst = Q + ((size_t)r * Hq + h) * hd;
  } else {
    const bool isk = h < Hq + Hkv;
    const int kvh = isk ? h - Hq : h - Hq - Hkv;
    if (cp >= 0) dst = (isk ? Kpool : Vpool) + kv_row_offset(g, seq, cp, kvh);
    else if (li >= 0) dst = (isk ? Kloc : Vloc) + ((size_t)li * Hkv + kvh) * hd;
  }
  float4 c = make_float4(0.f, 0.f, 0.f, 0.f), sv = c;
  if (rotate) { c = *reinterpret_cast<const float4 *>(cs + r * half + i); sv = *reinterpret_cast<const float4 *>(sn + r * half + i); }
#pragma unroll 1
  for (int walk = WALK ? 0 : 1; walk < 2; ++walk) {
    const bool live = !WALK || walk != 0;
    if (WALK && live) {
      pdl_wait();
      if (threadIdx.x == 0) tl_go(tl);
    }
    if (!mine) continue;
    const SLAB *p = live ? partials + (size_t)r * N + (size_t)h * hd + i : reinterpret_cast<const SLAB *>(cs);
    const size_t stride = live ? partial_stride : 0, half_at = live ? half : 0;
    float4 x1 = make_float4(0.f, 0.f, 0.f, 0.f), x2 = x1;
    // (both halves' loads together: two chains of additions)
#pragma unroll
    for (int s0 = 0; s0 < SLABS; s0 += 4) {
      if (s0 >= S) break;
      constexpr int AT_ONCE = SLABS < 4 ? SLABS : 4;
      float4 q1[AT_ONCE], q2[AT_ONCE];
#pragma unroll
      for (int t = 0; t < AT_ONCE; ++t)
        if (s0 + t < S) { q1[t] = load4<SLAB>(p + (s0 + t) * stride); q2[t] = load4<SLAB>(p + (s0 + t) * stride + half_at); }
#pragma unroll
      for (int t = 0; t < AT_ONCE; ++t)
        if (s0 + t < S) {
          x1.x += q1[t].x; x1.y += q1[t].y; x1.z += q1[t].z; x1.w += q1[t].w;
          x2.x += q2[t].x; x2.y += q2[t].y; x2.z += q2[t].z; x2.w += q2[t].w;
        }
    }
    if (bias) {
      const uint2 b1 = *reinterpret_cast<const uint2 *>(bias + (size_t)h * hd + i), b2 = *reinterpret_cast<const uint2 *>(bias + (size_t)h * hd + i + half);
      const float2 p0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&b1.x)), p1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&b1.y));
      const float2 q0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&b2.x)), q1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&b2.y));
      x1.x += p0.x; x1.y += p0.y; x1.z += p1.x; x1.w += p1.y;
      x2.x += q0.x; x2.y += q0.y; x2.z += q1.x; x2.w += q1.y;
    }
    if (hn) {
      // the upr = hd/8 threads of this head are consecutive lanes of one warp (upr is 8 or 16 and
      // divides the unit index), and all of them are here: the number of units is a multiple of upr
      float ss = x1.x * x1.x + x1.y * x1.y + x1.z * x1.z + x1.w * x1.w + x2.x * x2.x + x2.y * x2.y + x2.z * x2.z + x2.w * x2.w;
      const int lane = threadIdx.x & 31;
      const unsigned gmask = (upr >= 32 ? 0xffffffffu : ((1u << upr) - 1u)) << (lane & ~(upr - 1));
      for (int o = upr >> 1; o > 0; o >>= 1) ss += __shfl_xor_sync(gmask, ss, o);
      const float inv = rsqrtf(ss / (float)hd + eps);
      const uint2 g1 = *reinterpret_cast<const uint2 *>(hn + i), g2 = *reinterpret_cast<const uint2 *>(hn + i + half);
      const float2 p0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&g1.x)), p1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&g1.y));
      const float2 q0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&g2.x)), q1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&g2.y));
      x1.x *= inv * p0.x; x1.y *= inv * p0.y; x1.z *= inv * p1.x; x1.w *= inv * p1.y;
      x2.x *= inv * q0.x; x2.y *= inv * q0.y; x2.z *= inv * q1.x; x2.w *= inv * q1.y;
    }
    float4 y1 = x1, y2 = x2;
    if (rotate) {
      y1 = make_float4(x1.x * c.x - x2.x * sv.x, x1.y * c.y - x2.y * sv.y, x1.z * c.z - x2.z * sv.z, x1.w * c.w - x2.w * sv.w);
      y2 = make_float4(x2.x * c.x + x1.x * sv.x, x2.y * c.y + x1.y * sv.y, x2.z * c.z + x1.z * sv.z, x2.w * c.w + x1.w * sv.w);
    }
    __nv_bfloat162 a0 = __floats2bfloat162_rn(y1.x, y1.y), a1 = __floats2bfloat162_rn(y1.z, y1.w);
    __nv_bfloat162 b0 = __floats2bfloat162_rn(y2.x, y2.y), b1 = __floats2bfloat162_rn(y2.z, y2.w);
    uint2 o1, o2;
    o1.x = *reinterpret_cast<uint32_t *>(&a0); o1.y = *reinterpret_cast<uint32_t *>(&a1);
    o2.x = *reinterpret_cast<uint32_t *>(&b0); o2.y = *reinterpret_cast<uint32_t *>(&b1);
    if (live && dst) {
      *reinterpret_cast<uint2 *>(dst + i) = o1;
      *reinterpret_cast<uint2 *>(dst + i + half) = o2;
    }
  }
  if (threadIdx.x == 0) tl_end(tl);
}

// SwiGLU on an fp32 [R][2*ffn] projection whose columns interleave (gate_f, up_f).
__global__ void swiglu_kernel(const float *__restrict__ GU, int R, int ffn, bf16 *__restrict__ H) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (size_t)R * ffn) return;
  const float g = GU[2 * t], u = GU[2 * t + 1];
  H[t] = __float2bfloat16(g / (1.f + __expf(-g)) * u);
}

// SwiGLU over split-K slabs [S][R][ld] (fp32 or bf16) whose columns interleave (gate, up) and
// cover features [f0, f0 + nf): H[r][f0 + f] = silu(sum_s gate) * (sum_s up).  Two features per thread.
template <typename SLAB>
__global__ void swiglu_slab_kernel(const SLAB *__restrict__ slabs, int S, size_t stride, int R, int ld, int nf, int f0, int ldh,
                                   bf16 *__restrict__ H, TlSlot tl) {
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0) tl_go(tl);
  // two features per thread; silu with the fast division of the fused epilogue (a precise
  // division costs ~170 cycles per result and was most of this kernel's time)
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int nf2 = nf / 2;
  if (t >= (size_t)R * nf2) { if (threadIdx.x == 0) tl_end(tl); return; }
  const int r = (int)(t / nf2), f = (int)(t % nf2) * 2;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);                      // gate f, up f, gate f+1, up f+1
  add_slabs<4>(acc, slabs + (size_t)r * ld + 2 * f, S, stride);
  __nv_bfloat162 o = __floats2bfloat162_rn(__fdividef(acc.x, 1.f + __expf(-acc.x)) * acc.y, __fdividef(acc.z, 1.f + __expf(-acc.z)) * acc.w);
  *reinterpret_cast<__nv_bfloat162 *>(H + (size_t)r * ldh + f0 + f) = o;
  if (threadIdx.x == 0) tl_end(tl);
}

// Running per-row argmax over a chunk of logits [R][ncols] (fp32, leading dim ld)
// that covers vocabulary ids [col0, col0+ncols).  Lowest index wins ties; NaN never
// wins.  Optionally copies the chunk into a full [R][vocab] dump.
// With inv_temp > 0 the compared value is logit * inv_temp + Gumbel noise of (skey[r], id): a draw
// from softmax(logits / temperature) instead of the argmax; the dump always holds the raw logits.
__global__ void argmax_chunk_kernel(const float *__restrict__ L, int ld, int ncols, int col0, int first,
                                    float *__restrict__ best_val, int32_t *__restrict__ best_idx,
                                    float *__restrict__ dump, int vocab, float inv_temp, const uint32_t *__restrict__ skey) {
  const int r = blockIdx.x;
  float bv = -INFINITY; int bi = 0x7fffffff;
  const uint32_t key = inv_temp > 0.f ? skey[r] : 0u;
  for (int c = threadIdx.x; c < ncols; c += blockDim.x) {
    float v = L[(size_t)r * ld + c];
    if (dump) dump[(size_t)r * vocab + col0 + c] = v;
    if (inv_temp > 0.f) v = v * inv_temp + gumbel_noise(key, (uint32_t)(col0 + c));
    if (v > bv) { bv = v; bi = col0 + c; }
  }
  __shared__ float sv[32]; __shared__ int si[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, bv, o); const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
  }
  if ((threadIdx.x & 31) == 0) { sv[threadIdx.x >> 5] = bv; si[threadIdx.x >> 5] = bi; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
      if (sv[w] > bv || (sv[w] == bv && si[w] < bi)) { bv = sv[w]; bi = si[w]; }
    if (!first) {
      const float pv = best_val[r]; const int pi = best_idx[r];
      if (pv > bv || (pv == bv && pi < bi) || bi == 0x7fffffff) { bv = pv; bi = pi; }
    }
    if (bi == 0x7fffffff) bi = 0;
    best_val[r] = bv; best_idx[r] = bi;
  }
}

// Final argmax over the candidates [R][G] produced by the fused LM-head epilogue (one
// candidate per CTA and lane quadrant): one warp per row; a candidate index of -1 means
// "nothing valid".  Lowest index wins ties, which makes the result independent of the
// order in which candidates are combined.
__global__ void argmax_merge_kernel(const float *__restrict__ pv, const int32_t *__restrict__ pi, int G, int R,
                                    float *__restrict__ best_val, int32_t *__restrict__ best_idx, TlSlot tl) {
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0) tl_go(tl);
  const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (r >= R) { if (threadIdx.x == 0) tl_end(tl); return; }
  float bv = -INFINITY; int bi = 0x7fffffff;
  for (int g = lane; g < G; g += 32) {
    const float v = pv[(size_t)r * G + g]; const int i = pi[(size_t)r * G + g];
    if (i >= 0 && (v > bv || (v == bv && i < bi))) { bv = v; bi = i; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, bv, o); const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
  }
  if (lane == 0) { best_val[r] = bv; best_idx[r] = bi == 0x7fffffff ? 0 : bi; }
  if (threadIdx.x == 0) tl_end(tl);
}

// out[i] = sum over S slabs (fixed order) of in[s * stride + i].
__global__ void slab_sum_kernel(const float *__restrict__ in, int S, size_t stride, size_t n, float *__restrict__ out) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float v = 0.f;
  for (int s = 0; s < S; ++s) v += in[s * stride + i];
  out[i] = v;
}

// ---------------------------------------------------------------------------
// Draft / verify / select (paper Section 3.2; Section 4.4.3).
// One warp per sequence, lane i = causal slot i:
//   target_i = verified prediction for position n+i+1: argmax of causal slot i's logits, or
//              (tgt_ids != null) the argmax of the row that mixes them with the first slot
//              of block i;
//   draft i >= 1 agrees iff the sequence had a draft there (i < blk_len) and
//              block[i] == target_{i-1};
//   L = 1 + length of the leading run of agreeing drafts (slot 0 is settled), or the
//   forced value;  emitted = block[1..L-1], target_{L-1};
//   next block = target_{L-1}, then the argmax of mask slots (L-1, 1..k-1); with no mask
//   blocks (plain autoregressive step, k = 1) the next block is target_0 alone.
// Commits as well (paper Section 3.3): the causal slots' K/V are in the cache at n..n+k-1, committing L of them is
// n <- n + L.  The last block to finish closes the step: it moves the turn on and leaves turn number and status with the results.
// ---------------------------------------------------------------------------
__global__ void verify_select_kernel(const int32_t *__restrict__ arg_ids, const int32_t *__restrict__ tgt_ids,
                                     const int32_t *__restrict__ step_seqs,
                                     const int32_t *__restrict__ forced, int k, int n_blocks, StepLayout lay, int k_max,
                                     int32_t *__restrict__ block_ids, int32_t *__restrict__ blk_len, const int32_t *__restrict__ step_n,
                                     int32_t *__restrict__ step_L, int32_t *__restrict__ seq_len, StepIo io, TlSlot tl) {
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0) tl_go(tl);
  const int s = blockIdx.x, lane = threadIdx.x;
  const int turn = *io.turn;
  int32_t *out = io.out[turn & 1];                // [n_seqs][k_max+1]
  if (lay.k) { k = lay.k[s]; n_blocks = k; }
  const int T = k * (n_blocks + 1);
  const int seq = step_seqs[s];
  const int32_t *ids = arg_ids + (lay.k ? (size_t)lay.off[s] : (size_t)s * T);
  int32_t *blk = block_ids + (size_t)seq * k_max;
  const int valid = blk_len[seq];
  size_t tgt0 = (size_t)s * k;                    // this sequence's first verification target among the mixed rows
  if (lay.k && tgt_ids) { tgt0 = 0; for (int t = 0; t < s; ++t) tgt0 += lay.k[t]; }
  const int tgt = lane < k ? (tgt_ids ? tgt_ids[tgt0 + lane] : ids[lane]) : -1;
  const int mine = lane < k ? (lane < valid ? blk[lane] : -2) : -2;
  const int prev_tgt = __shfl_up_sync(0xffffffffu, tgt, 1);
  const bool agree = lane == 0 || (lane < k && lane < valid && mine == prev_tgt);
  const unsigned bits = __ballot_sync(0xffffffffu, agree);
  int L = __ffs(~bits) - 1;            // leading run of ones; bit 0 is always set
  if (L > k || L < 0) L = k;           // all 32 lanes agreeing gives ffs(0) = 0
  const int f = forced ? forced[s] : 0;
  if (f > 0) L = f;
  const int t_last = __shfl_sync(0xffffffffu, tgt, L - 1);
  const int next_draft = (n_blocks > 0 && lane >= 1 && lane < k) ? ids[k + (L - 1) * k + lane] : 0;
  const int shifted = __shfl_down_sync(0xffffffffu, mine, 1);     // block[lane+1]
  __syncwarp();
  if (lane < k) {
    out[(size_t)s * (k_max + 1) + 1 + lane] = lane < L - 1 ? shifted : (lane == L - 1 ? t_last : -1);
    blk[lane] = lane == 0 ? t_last : next_draft;
  }
  if (lane == 0) { out[(size_t)s * (k_max + 1)] = L; step_L[s] = L; seq_len[seq] = step_n[s] + L; blk_len[seq] = n_blocks > 0 ? k : 1; tl_end(tl); }
  __threadfence_system();
  __syncwarp();
  if (lane == 0 && atomicAdd(io.blocks_done, 1) == (int)gridDim.x - 1) {
    *io.blocks_done = 0; *io.turn = turn + 1;
    volatile int32_t *done = io.done[turn & 1];
    done[1] = *(volatile int32_t *)io.status;
    __threadfence_system();
    done[0] = turn + 1;
  }
}

// Verification by a mix of the autoregressive and the diffusion prediction (paper Section 4.4.3:
// argmax(beta * logits_ar + (1 - beta) * logits_diff)).  Logits are linear in the final-normed
// hidden row, so the mix is taken there: row dst = beta * row a + (1 - beta) * row b of the LM
// head's input, one extra input row per verified position, and the LM head's argmax of that row
// is the argmax of the mixed logits.  Block i handles pair i:
//   a = a0 + (i / k) * a_seq + (i % k) * a_j,  b likewise,  dst = dst0 + i.
// With per-sequence block lengths (lay.k != null) pair i belongs to the sequence whose pairs
// (one per verified position, k_s of them) contain it: a = off_s + j, b = off_s + k_s + j * k_s.
__global__ void mix_rows_kernel(bf16 *__restrict__ A, int d, float beta, int k, int a0, int a_seq, int a_j, int b0, int b_seq, int b_j,
                                StepLayout lay, int dst0, uint32_t *__restrict__ skey, TlSlot tl) {
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0) tl_go(tl);
  const int i = blockIdx.x;
  int row_a, row_b;
  if (lay.k) {
    int s = 0, p = 0;
    while (s + 1 < lay.n_seqs && i >= p + lay.k[s]) { p += lay.k[s]; ++s; }
    const int ks = lay.k[s], j = i - p;
    row_a = lay.off[s] + j; row_b = lay.off[s] + ks + j * ks;
  } else {
    const int s = i / k, j = i % k;
    row_a = a0 + s * a_seq + j * a_j; row_b = b0 + s * b_seq + j * b_j;
  }
  const bf16 *ra = A + (size_t)row_a * d, *rb = A + (size_t)row_b * d;
  bf16 *ro = A + (size_t)(dst0 + i) * d;
  if (skey && threadIdx.x == 0) skey[dst0 + i] = skey[row_a];     // the mixed row predicts what row a predicts
  for (int c = threadIdx.x * 2; c < d; c += blockDim.x * 2) {
    const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(ra + c));
    const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(rb + c));
    *reinterpret_cast<__nv_bfloat162 *>(ro + c) = __floats2bfloat162_rn(beta * x.x + (1.f - beta) * y.x, beta * x.y + (1.f - beta) * y.y);
  }
  if (threadIdx.x == 0) tl_end(tl);
}

// Running log-sum-exp of a row over vocabulary chunks, and the logit of the row's target id.
// L [R][ld] holds the logits of ids [col0, col0 + ncols).  (run_max, run_sum) is updated so that
// log sum_v exp(logit_v) = run_max + log(run_sum) after the last chunk; fixed reduction order.
__global__ void __launch_bounds__(256)
score_chunk_kernel(const float *__restrict__ L, int ld, int ncols, int col0, int first, const int32_t *__restrict__ target,
                   float *__restrict__ run_max, float *__restrict__ run_sum, float *__restrict__ tgt_logit) {
  __shared__ float red[8];
  __shared__ float bcast;
  const int r = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float *row = L + (size_t)r * ld;
  float m = -INFINITY;
  for (int c = threadIdx.x; c < ncols; c += 256) m = fmaxf(m, row[c]);
  m = warp_max(m);
  if (lane == 0) red[warp] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = red[0];
    for (int i = 1; i < 8; ++i) t = fmaxf(t, red[i]);
    bcast = first ? t : fmaxf(t, run_max[r]);
  }
  __syncthreads();
  const float M = bcast;
  float sum = 0.f;
  for (int c = threadIdx.x; c < ncols; c += 256) sum += __expf(row[c] - M);
  sum = warp_sum(sum);
  __syncthreads();
  if (lane == 0) red[warp] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int i = 0; i < 8; ++i) t += red[i];
    if (!first) t += run_sum[r] * __expf(run_max[r] - M);
    run_max[r] = M; run_sum[r] = t;
    const int tg = target[r] - col0;
    if (tg >= 0 && tg < ncols) tgt_logit[r] = row[tg];
  }
}

// logprob[r] = tgt_logit[r] - (run_max[r] + log(run_sum[r]))
__global__ void score_finish_kernel(const float *__restrict__ run_max, const float *__restrict__ run_sum, const float *__restrict__ tgt_logit,
                                    int R, float *__restrict__ logprob) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < R) logprob[r] = tgt_logit[r] - (run_max[r] + logf(run_sum[r]));
}

// The same from per-group (max, sum) pairs [parts][R]; 16 rows per block, 32 threads share a row's groups (fixed order).
__global__ void __launch_bounds__(512)
score_merge_kernel(const float2 *__restrict__ lse, int parts, const float *__restrict__ tgt_logit, int R, float *__restrict__ logprob) {
  __shared__ float2 red[32][16];
  const int i = threadIdx.x & 15, sub = threadIdx.x >> 4, r = blockIdx.x * 16 + i;
  float M = -INFINITY, sum = 0.f;
  pdl_wait();
  if (r < R) {
    for (int p0 = sub; p0 < parts; p0 += 32 * 8) {
      float2 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = p0 + u * 32 < parts ? lse[(size_t)(p0 + u * 32) * R + r] : make_float2(-INFINITY, 0.f);
      float m = M;
#pragma unroll
      for (int u = 0; u < 8; ++u) m = fmaxf(m, v[u].x);
      const float ref = m == -INFINITY ? 0.f : m;
      sum *= __expf(M - ref);
#pragma unroll
      for (int u = 0; u < 8; ++u) sum += v[u].y * __expf(v[u].x - ref);
      M = m;
    }
  }
  red[sub][i] = make_float2(M, sum);
  __syncthreads();
  if (sub == 0 && r < R) {
    for (int s = 1; s < 32; ++s) M = fmaxf(M, red[s][i].x);
    sum = 0.f;
    for (int s = 0; s < 32; ++s) sum += red[s][i].y * __expf(red[s][i].x - M);
    logprob[r] = tgt_logit[r] - (M + logf(sum));
  }
}

// First-pass finish: settled token = argmax of the last prompt row; drafts = argmax
// of mask rows 1..k-1 (paper Section 3.2, start of generation).
// row_first: the row whose argmax is the settled token (the last prompt row, or the extra row that
// mixes it with the first mask row when beta < 1).
__global__ void prefill_finish_kernel(const int32_t *__restrict__ arg_ids, int row_last_prompt, int row_first, int k, int k_max, int seq,
                                      int n_prompt, int32_t *__restrict__ block_ids, int32_t *__restrict__ blk_len,
                                      int32_t *__restrict__ seq_len, const int32_t *status, int32_t *out /*pinned: first token, status*/) {
  const int i = threadIdx.x;
  if (i < k) block_ids[(size_t)seq * k_max + i] = i == 0 ? arg_ids[row_first] : arg_ids[row_last_prompt + 1 + i];
  if (i == 0) { seq_len[seq] = n_prompt; blk_len[seq] = k; out[0] = arg_ids[row_first]; out[1] = *(volatile const int32_t *)status; }
}

// ---------------------------------------------------------------------------
// KV eviction check (debug): after a step has committed L of its k causal slots, positions n+L..n+k-1 are dead and
// get overwritten by the next step.  This fills them, in every layer, with the
// largest finite bf16 (3.4e38), so that any later use of evicted data with a non-zero
// weight would surface as inf/NaN or a wild value.  (Not NaN itself: the tensor-core
// attention loads whole 64-position pages and multiplies the masked positions' V rows
// by an exact zero, which must stay zero.)  Grid (n_seqs, n_layers).
// ---------------------------------------------------------------------------
__global__ void kv_poison_kernel(const int32_t *__restrict__ step_seqs, const int32_t *__restrict__ step_n, const int32_t *__restrict__ step_L, int k,
                                 const int32_t *__restrict__ step_k, KvGeom g, bf16 *__restrict__ kv_base, size_t pool_stride, TlSlot tl) {
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0) tl_go(tl);
  const int s = blockIdx.x, l = blockIdx.y;
  if (step_k) k = step_k[s];
  const int seq = step_seqs[s];
  const int n = step_n[s], L = step_L[s];
  bf16 *Kp = kv_base + (size_t)(2 * l) * pool_stride, *Vp = Kp + pool_stride;
  const int per = g.n_kv_heads * g.head_dim;
  const bf16 nanv = __ushort_as_bfloat16((unsigned short)0x7f7f);
  for (int t = threadIdx.x; t < (k - L) * per; t += blockDim.x) {
    const int p = n + L + t / per, kvh = (t % per) / g.head_dim, c = t % g.head_dim;
    const size_t off = kv_row_offset(g, seq, p, kvh) + c;
    Kp[off] = nanv; Vp[off] = nanv;
  }
  if (threadIdx.x == 0) tl_end(tl);
}

// Gather cached K/V rows into canonical [npos][Hkv][hd] order (debug read-back).
__global__ void kv_gather_kernel(const bf16 *__restrict__ Kp, const bf16 *__restrict__ Vp, KvGeom g, int seq, int pos0,
                                 bf16 *__restrict__ ko, bf16 *__restrict__ vo) {
  const int p = blockIdx.x, kvh = blockIdx.y;
  const size_t off = kv_row_offset(g, seq, pos0 + p, kvh);
  for (int c = threadIdx.x; c < g.head_dim; c += blockDim.x) {
    ko[((size_t)p * g.n_kv_heads + kvh) * g.head_dim + c] = Kp[off + c];
    vo[((size_t)p * g.n_kv_heads + kvh) * g.head_dim + c] = Vp[off + c];
  }
}

// Probe of the bounded wait every tensor-core kernel is built on: one thread waits, with a
// short limit, on an mbarrier that nothing will ever arrive on, gives up, and reports it through
// the status word, exactly as a kernel whose producer went missing would.  Nothing hangs: the
// wait is the same bounded loop, only shorter.  waited[0] receives the polls it took.
__global__ void wait_probe_kernel(uint32_t limit, int *status, int *waited) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    sm100::mbar_init(sm100::smem_u32(&bar), 1);
    sm100::fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const bool ok = sm100::mbar_wait(sm100::smem_u32(&bar), 0u, &abort_flag, limit);      // phase 0 never completes
    waited[0] = ok ? 0 : (int)limit;
    if (!ok && abort_flag) atomicExch(status, 9);
  }
}
