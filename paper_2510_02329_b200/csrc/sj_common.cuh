// Shared device-side definitions for the verification-step kernels (sm_100a).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace sj {

typedef __nv_bfloat16 bf16;

constexpr int kMaxBatch = 256;
constexpr int kMaxGamma = 31;
constexpr int kMaxRows = 512;
constexpr int kTileN = 128;  // output features per GEMM tile (the MMA's M after swapping operands)

// device status word values (first error wins)
enum DevStatus { DEV_OK = 0, DEV_TIMEOUT = 7, DEV_STATE = 3 };

__device__ __forceinline__ float to_f(float x) { return x; }
__device__ __forceinline__ float to_f(bf16 x) { return __bfloat162float(x); }
template <typename T> __device__ __forceinline__ T from_f(float x);
template <> __device__ __forceinline__ float from_f<float>(float x) { return x; }
template <> __device__ __forceinline__ bf16 from_f<bf16>(float x) { return __float2bfloat16_rn(x); }

// Per-call arguments, resident in device memory and rewritten by k_begin at the start of a call so
// that a captured graph never bakes in a caller's pointer.
struct StepArgs {
  const int* draft_ids;
  const float* q_tok;
  const float* q_full;
  const float* uniforms;
  int* accepted_len;
  int* next_token;
  float* judge_scores;
  float* p_draft;
  int* new_kv_len;
  float* dbg_hidden;
  float* dbg_logits;
  float* logp_draft;      // optional: natural log of p_j(d_j)
  int B, gamma, mode, use_align, use_judge, commit;
  int top_k;              // greedy alignment test: the draft must be among the target's top_k tokens (1 or 2)
  int accept_all;         // every drafted position is accepted whatever the tests say (prefill, teacher forcing)
  // A block that continues itself (prefill): entry b of the batch is the next `pos_step` rows of the same sequence, so
  // its cache is pos_step * b tokens longer than the stored length, and row r's input token is row_tok[r] (r < n_tok;
  // null: the pending token and the drafts).  0 and null in a verification step.
  const int* row_tok;
  int n_tok, pos_step;
  int kv_rows;            // rows r >= kv_rows store no key / value rows in the pages (padding rows; blocks only scored)
  float inv_temperature, judge_bias;
  int has_judge;
  int seq_ids[kMaxBatch];
  float theta[kMaxBatch]; // judge threshold per sequence of the batch
};

// Paged KV cache view.  Element (layer, page, kv in {0,1}, head, slot, dim):
//   pool[((((layer * n_pages + page) * 2 + kv) * Hkv + head) * page_size + slot) * hd + dim]
struct KvView {
  void* pool;
  int* block_table;        // [max_seqs, max_pages_per_seq]
  int* kv_len;             // [max_seqs]
  int* pending;            // [max_seqs]
  long n_pages;
  int max_pages_per_seq;
  int page_size;           // 16
  int n_kv_heads, head_dim;
};

template <typename T>
__device__ __forceinline__ T* kv_row(const KvView& kv, int layer, int page, int which, int head, int slot) {
  size_t idx = ((((size_t)layer * kv.n_pages + page) * 2 + which) * kv.n_kv_heads + head);
  idx = (idx * kv.page_size + slot) * kv.head_dim;
  return reinterpret_cast<T*>(kv.pool) + idx;
}

// Changes of a cache's bookkeeping.  They travel as kernel parameters, one launch for all sequences, instead of as a copy
// from host memory per sequence.
struct KvEdit { int seq, at, value; };   // at >= 0: entry of the block table; else one of:
constexpr int kEditLen = -1, kEditPending = -2, kMaxEdits = kMaxBatch;
struct KvEdits { int n; KvEdit e[kMaxEdits]; };

// How a GEMM's output tile is spread over thread blocks (split along K).  Work is counted in
// units of (128-feature tile, 64-wide K block) -- fp32 models (64, 128) --; block c owns units [c*U/G, (c+1)*U/G).  A tile's
// partial sums live in consecutive "slots" of the partial buffer, one per contributing block in
// block order, so that the consumer adds them in a fixed order (no atomics, bit-reproducible).
struct SplitPlan {
  const int2* tile_slots;  // per tile: (first contributing block, number of slots); null: one slot
  int n_tiles;
  int tile_shift;          // log2 of a tile's features
};

// Partial buffer layout: P[slot][row][N] fp32.
__device__ __forceinline__ float reduce_partials(const float* __restrict__ P, const SplitPlan& sp, size_t slot_stride,
                                                 int N, int r, int n) {
  const float* p = P + (size_t)r * N + n;
  if (sp.tile_slots == nullptr) return *p;
  const int cnt = sp.tile_slots[n >> sp.tile_shift].y;
  float s = 0.f;
  for (int i = 0; i < cnt; i += 4) {   // four slots in flight, added in order
    float v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = p[(size_t)min(i + u, cnt - 1) * slot_stride];
#pragma unroll
    for (int u = 0; u < 4; ++u) s += i + u < cnt ? v[u] : 0.f;
  }
  return s;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Sums of N values (N = 4, 8 or 16) over the 32 lanes of a warp, all at once: every exchange halves the values a lane
// still carries (16 shuffles for N = 16 instead of 80).  A lane returns the total of value lane / (32 / N).
template <int N>
__device__ __forceinline__ float warp_sum_n(const float* v, int lane) {
  float a[N];
#pragma unroll
  for (int i = 0; i < N; ++i) a[i] = v[i];
  int bit = 16;
#pragma unroll
  for (int h = N / 2; h >= 1; h >>= 1, bit >>= 1) {
    const bool up = lane & bit;
#pragma unroll
    for (int i = 0; i < h; ++i) a[i] = (up ? a[i + h] : a[i]) + __shfl_xor_sync(0xffffffffu, up ? a[i] : a[i + h], bit);
  }
#pragma unroll
  for (; bit >= 1; bit >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], bit);
  return a[0];
}
// The same for the maximum of value i over the warp, with the lowest `id` among the lanes that have it.
template <int N>
__device__ __forceinline__ void warp_max_n(const float* v, int id, int lane, float& m, int& arg) {
  float a[N];
  int b[N];
#pragma unroll
  for (int i = 0; i < N; ++i) { a[i] = v[i]; b[i] = id; }
  int bit = 16;
#pragma unroll
  for (int h = N / 2; h >= 1; h >>= 1, bit >>= 1) {
    const bool up = lane & bit;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float mine = up ? a[i + h] : a[i], om = __shfl_xor_sync(0xffffffffu, up ? a[i] : a[i + h], bit);
      const int mid = up ? b[i + h] : b[i], oid = __shfl_xor_sync(0xffffffffu, up ? b[i] : b[i + h], bit);
      const bool take = om > mine || (om == mine && oid < mid);
      a[i] = take ? om : mine;
      b[i] = take ? oid : mid;
    }
  }
#pragma unroll
  for (; bit >= 1; bit >>= 1) {
    const float om = __shfl_xor_sync(0xffffffffu, a[0], bit);
    const int oid = __shfl_xor_sync(0xffffffffu, b[0], bit);
    const bool take = om > a[0] || (om == a[0] && oid < b[0]);
    a[0] = take ? om : a[0];
    b[0] = take ? oid : b[0];
  }
  m = a[0];
  arg = b[0];
}

// Maximum of each of N values (N = 8 or 16) over the warp: a lane returns that of value lane / (32 / N).
template <int N>
__device__ __forceinline__ float warp_fmax_n(const float* v, int lane) {
  float a[N];
#pragma unroll
  for (int i = 0; i < N; ++i) a[i] = v[i];
  int bit = 16;
#pragma unroll
  for (int h = N / 2; h >= 1; h >>= 1, bit >>= 1) {
    const bool up = lane & bit;
#pragma unroll
    for (int i = 0; i < h; ++i) a[i] = fmaxf(up ? a[i + h] : a[i], __shfl_xor_sync(0xffffffffu, up ? a[i] : a[i + h], bit));
  }
#pragma unroll
  for (; bit >= 1; bit >>= 1) a[0] = fmaxf(a[0], __shfl_xor_sync(0xffffffffu, a[0], bit));
  return a[0];
}

// Block-wide sum with a fixed reduction tree (deterministic).  `red` holds >= 32 floats.
__device__ __forceinline__ float block_sum(float v, float* red) {
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  float t = (threadIdx.x < nw) ? red[threadIdx.x] : 0.f;
  if (w == 0) {
    t = warp_sum(t);
    if (lane == 0) red[0] = t;
  }
  __syncthreads();
  return red[0];
}

// Programmatic dependent launch: every kernel of the step calls pdl_wait() before it reads or
// writes anything another kernel of the step produces, and pdl_launch() once its own dependents
// may be scheduled.  Both are no-ops when the launch carries no programmatic dependency.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Softmax statistics of a set of logits: running maximum m, sum of exp(z - m), arg max.
struct RowStat {
  float m, s;
  int arg;
  int pad;   // top-k test: how many of the set's logits rank before the drafted token's (larger, or equal with a lower id)
};
__device__ __forceinline__ RowStat stat_merge(const RowStat& a, const RowStat& b) {
  // a precedes b in vocabulary order: on equal maxima the lower index (a) is kept
  RowStat r;
  bool take_b = b.m > a.m;
  r.m = take_b ? b.m : a.m;
  r.arg = take_b ? b.arg : a.arg;
  float sa = (a.m == -INFINITY) ? 0.f : a.s * expf(a.m - r.m);
  float sb = (b.m == -INFINITY) ? 0.f : b.s * expf(b.m - r.m);
  r.s = sa + sb;
  r.pad = a.pad + b.pad;
  return r;
}

// The same for sets in any vocabulary order: on equal maxima the lower index is kept.
__device__ __forceinline__ RowStat stat_merge_any(const RowStat& a, const RowStat& b) {
  return (b.m == a.m && b.arg < a.arg) ? stat_merge(b, a) : stat_merge(a, b);
}

// Merged statistics of the block rows [r0, r0 + rows) over all vocabulary tiles, by the eight warps of a block: a warp
// takes half of a row's tiles, 16 of them per lane in flight (a thread walking through its tiles one load at a time took
// 4 us a row, 60 us of a 9-row step in all).  part: [rows][2], shared memory; the caller synchronises and merges the halves
// with merge_row_halves().
__device__ __forceinline__ void merge_row_stats(const RowStat* stats, int n_vtiles, int R, int r0, int rows, int warp, int lane,
                                                RowStat (*part)[2]) {
  const int half = (n_vtiles + 1) / 2;
#pragma unroll 1
  for (int item = warp; item < 2 * rows; item += 8) {
    const int j = item >> 1, t0 = (item & 1) * half, t1 = min(t0 + half, n_vtiles);
    RowStat a; a.m = -INFINITY; a.s = 0.f; a.arg = 0x7fffffff; a.pad = 0;
#pragma unroll 1
    for (int tb = t0; tb < t1; tb += 512) {
      float4 raw[16];
#pragma unroll
      for (int k = 0; k < 16; ++k)
        raw[k] = __ldcg(reinterpret_cast<const float4*>(stats + (size_t)min(tb + 32 * k + lane, t1 - 1) * R + r0 + j));
      float m = -INFINITY, sum = 0.f;
      int arg = 0x7fffffff;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        if (tb + 32 * k + lane >= t1) { raw[k].x = -INFINITY; raw[k].z = __int_as_float(0x7fffffff); raw[k].w = 0.f; }
        const int ak = __float_as_int(raw[k].z);
        if (raw[k].x > m || (raw[k].x == m && ak < arg)) { m = raw[k].x; arg = ak; }
      }
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        sum += raw[k].x == -INFINITY ? 0.f : raw[k].y * expf(raw[k].x - m);
        a.pad += __float_as_int(raw[k].w);
      }
      RowStat b; b.m = m; b.s = sum; b.arg = arg; b.pad = 0;
      a = stat_merge_any(a, b);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      RowStat b;
      b.m = __shfl_xor_sync(0xffffffffu, a.m, o);
      b.s = __shfl_xor_sync(0xffffffffu, a.s, o);
      b.arg = __shfl_xor_sync(0xffffffffu, a.arg, o);
      b.pad = __shfl_xor_sync(0xffffffffu, a.pad, o);
      a = stat_merge_any(a, b);
    }
    if (lane == 0) part[j][item & 1] = a;
  }
}

__device__ __forceinline__ RowStat merge_row_halves(const RowStat (&part)[2]) {
  RowStat a = stat_merge_any(part[0], part[1]);
  if (a.arg == 0x7fffffff) a.arg = 0;   // no logit is larger than -infinity (all are NaN): a token of the vocabulary all the same
  return a;
}

}  // namespace sj
