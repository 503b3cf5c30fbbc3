// Elementwise, CUDA-core GEMM / attention, LM-head statistics and acceptance kernels of the
// verification step.  Templated on the storage type T (float or bf16); accumulation is fp32.
#pragma once

#include "sj_common.cuh"

namespace sj {

// Device workspace of one target (all sized for max_rows).
struct Work {
  float* X;          // [R, d]        fp32 residual stream
  // GEMM inputs.  fp32 models: one plane [R, K] of floats.  bf16 models: TWO bf16 planes
  // [2][Rp][K] (Rp = R rounded up to 16): plane 0 holds bf16(x), plane 1 holds bf16(x - plane 0), so
  // that the tensor cores see x to ~2^-17 instead of 2^-9; the product with both planes is summed
  // in the fp32 accumulator's epilogue.
  void* A;           // normalised activations (input of QKV / gate-up / LM head), K = d
  float* Q;          // [R, Hq*hd]    fp32 rotated queries
  __half* Qb;        // [B, Hkv, group*(gamma+1), hd] fp16 rotated queries times log2(e)/sqrt(hd), query row
                     // g*(gamma+1)+j of a KV head's group (tensor-core attention), or null
  __half* Qlo;       // same layout: what the fp16 rounding of Qb dropped (q - Qb, rounded to fp16), for the layers in
                     // which the attention runs with two-term operands
  __half* KVn;       // [B, Hkv, 2 (K|V), gamma+1, hd] fp16 copy of this step's own key / value rows (the rows the
                     // pages receive in bf16): the tensor-core attention reads the block's own rows from here
  void* ATT;         // attention output (input of the O projection), K = Hq*hd
  void* H;           // silu(gate)*up (input of the down projection), K = F
  float* P;          // partial sums of the current GEMM: [slot][R][N]
  float* ssq;        // [2][d / 128][R] sums of squares of the residual rows per 128 columns (wide steps: input of QKV, of
                     // gate/up)
  float* Hf;         // [R, d]        fp32 hidden state after the final norm
  float2* rope;      // [R, hd/2]     (cos, sin) of this step's positions
  int* row_pos;      // [R]           absolute position of each row
  int* chunk_start;  // [B+1]         prefix sum of attention chunks per sequence
  float* att_m;      // [chunks, Hq, gamma+1]         running max of each partial
  float* att_l;      // same                           sum of exp
  float* att_o;      // [chunks, Hq, gamma+1, hd]      unnormalised partial outputs
  float* tc_m;       // tensor-core attention partials: [slots][4][nq] running max (log2 domain)
  float* tc_l;       // same                            sum of exp2
  float* tc_o;       // [slots][4][nq][hd]              unnormalised outputs
  RowStat* stats;    // [vocab tiles, R]
  float* tgt_logit;  // [R]   logit of the drafted token d_{j+1} in row j
  float* tgt_pre;    // [R]   the same logit (raw), computed BEFORE the LM head when the top-k test needs it to count ranks
  RowStat* rowstat;  // [R]   merged statistics
  float* logits;     // [R, V] fp32, or null: stored for the CUDA-core LM head and in sampling mode (the row that a token is
                     // drawn from is known only after the head); may be P
  void* Asel;        // GEMM input planes of one row (the last of a prefill), K = d
  double2* rs_part;  // [B][chunks of the vocabulary] sums of p and max(0, p - q) of the row that is drawn from
  const double* inv_freq;  // [hd/2] rope_theta^(-2i/hd)
  const float* judge_w;    // [d]
  int* status;
};

struct Dims {
  int n_layers, d, Hq, Hkv, hd, F, V;
  float eps;
};

__host__ __device__ __forceinline__ int pad16(int r) { return (r + 15) & ~15; }

// Store one GEMM-input element (row r of R, column i of K).
template <typename T> __device__ __forceinline__ void store_act(void* base, int R, int K, int r, int i, float y);
template <> __device__ __forceinline__ void store_act<float>(void* base, int R, int K, int r, int i, float y) {
  reinterpret_cast<float*>(base)[(size_t)r * K + i] = y;
}
template <> __device__ __forceinline__ void store_act<bf16>(void* base, int R, int K, int r, int i, float y) {
  bf16 hi = __float2bfloat16_rn(y);
  bf16 lo = __float2bfloat16_rn(y - __bfloat162float(hi));
  bf16* b = reinterpret_cast<bf16*>(base);
  b[(size_t)r * K + i] = hi;
  b[((size_t)pad16(R) + r) * K + i] = lo;
}

// ---------------------------------------------------------------------------------------------
// step set-up
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void apply_edits(const KvView& kv, const KvEdits& edits, int tid, int nthreads) {
  for (int i = tid; i < edits.n; i += nthreads) {
    const KvEdit e = edits.e[i];
    if (e.at >= 0) kv.block_table[(size_t)e.seq * kv.max_pages_per_seq + e.at] = e.value;
    else (e.at == kEditLen ? kv.kv_len : kv.pending)[e.seq] = e.value;
  }
}
static __global__ void k_edit(KvView kv, const __grid_constant__ KvEdits edits) { apply_edits(kv, edits, threadIdx.x, blockDim.x); }

// The start of a call: its arguments go to device memory (d_args), its new pages into the block table.  Per-stage steps
// (plan): row positions and the attention chunk list, from the true cache lengths; the persistent kernel: its barrier
// counter and abort word (sync, four words) back to zero.  One launch with everything in its parameters, in place of two or
// more copies, a memset and a set-up kernel: a step of the toy model 55.8 -> 51.1 us (B200; steps of a millisecond, whose copies
// the stream takes in its stride, are the same).
static __global__ void k_begin(const __grid_constant__ StepArgs a, const __grid_constant__ KvEdits edits, StepArgs* __restrict__ d_args, KvView kv,
                               Work w, int chunk_len, int plan, unsigned* __restrict__ sync) {
  pdl_launch();
  __shared__ int nch[kMaxBatch];
  static_assert(sizeof(StepArgs) % 4 == 0, "copied word by word");
  for (int i = threadIdx.x; i < (int)(sizeof(StepArgs) / 4); i += blockDim.x)
    reinterpret_cast<int*>(d_args)[i] = reinterpret_cast<const int*>(&a)[i];
  apply_edits(kv, edits, threadIdx.x, blockDim.x);
  if (sync && threadIdx.x < 4) sync[threadIdx.x] = 0u;
  if (!plan) return;
  const int B = a.B, rows = a.gamma + 1;
  for (int b = threadIdx.x; b < B; b += blockDim.x) {
    const int L = kv.kv_len[a.seq_ids[b]] + b * a.pos_step;
    nch[b] = (L + rows + chunk_len - 1) / chunk_len;
    for (int j = 0; j < rows; ++j) w.row_pos[b * rows + j] = L + j;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int b = 0; b < B; ++b) {
      w.chunk_start[b] = acc;
      acc += nch[b];
    }
    w.chunk_start[B] = acc;
  }
}

// RMSNorm of a row held in shared memory; writes T activations and optional fp32 copies.
template <typename T>
__device__ __forceinline__ void norm_row_from_smem(const float* xs, int d, const T* __restrict__ gain, float eps,
                                                   void* act, int R, int r, float* hf_row, float* dbg_row, float* red) {
  float ss = 0.f;
  for (int i = threadIdx.x; i < d; i += blockDim.x) ss += xs[i] * xs[i];
  ss = block_sum(ss, red);
  float inv = 1.0f / sqrtf(ss / (float)d + eps);
  for (int i = threadIdx.x; i < d; i += blockDim.x) {
    float y = xs[i] * inv * to_f(gain[i]);
    store_act<T>(act, R, d, r, i, y);
    if (hf_row) hf_row[i] = y;
    if (dbg_row) dbg_row[i] = y;
  }
}

// a1 + first a2: embedding gather, RMSNorm, and this step's rotary table.  With `ssq` ([d / 128][R]; the paired projections,
// whose d is a multiple of 128) the planes hold embedding x gain and the reader applies the row scalar, as in the other
// layers and in the persistent kernel: a product of two bf16 numbers fits the two planes, so the first layer's keys and
// values carry no activation rounding.  Normalised rows lose 2^-17 in the planes, which turned the bf16 rounding of 2.5e-3 of
// the first layer's cached numbers (6.5e-4 without it, 8e-4 by the persistent kernel), and of more in every layer after.
template <typename T>
__global__ void k_embed_norm(const StepArgs* __restrict__ args, KvView kv, Work w, Dims dm, const T* __restrict__ embed,
                             const T* __restrict__ gain, float* __restrict__ ssq) {
  extern __shared__ float xs[];
  __shared__ float red[32];
  pdl_wait();
  pdl_launch();
  const int r = blockIdx.x, rows = args->gamma + 1;
  const int b = r / rows, j = r % rows;
  const int seq = args->seq_ids[b];
  int tok;
  if (args->row_tok) tok = args->row_tok[min(r, args->n_tok - 1)];
  else tok = (j == 0) ? kv.pending[seq] : args->draft_ids[b * args->gamma + j - 1];
  tok = min(max(tok, 0), dm.V - 1);
  const T* e = embed + (size_t)tok * dm.d;
  for (int i = threadIdx.x; i < dm.d; i += blockDim.x) {
    float x = to_f(e[i]);
    xs[i] = x;
    w.X[(size_t)r * dm.d + i] = x;
  }
  const int pos = kv.kv_len[seq] + b * args->pos_step + j;
  for (int i = threadIdx.x; i < dm.hd / 2; i += blockDim.x) {
    double s, c;
    sincos((double)pos * w.inv_freq[i], &s, &c);
    w.rope[(size_t)r * (dm.hd / 2) + i] = make_float2((float)c, (float)s);
  }
  __syncthreads();
  if (ssq) {   // uniform
    const int lane = threadIdx.x & 31;
    for (int t = threadIdx.x >> 5; t < dm.d / 128; t += blockDim.x >> 5) {
      float ss = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int f = t * 128 + 32 * i + lane;
        const float x = xs[f];
        store_act<T>(w.A, gridDim.x, dm.d, r, f, x * to_f(gain[f]));
        ss += x * x;
      }
      ss = warp_sum(ss);
      if (lane == 0) ssq[(size_t)t * gridDim.x + r] = ss;
    }
    return;
  }
  norm_row_from_smem<T>(xs, dm.d, gain, dm.eps, w.A, gridDim.x, r, nullptr, nullptr, red);
}

// a6/a8 tail + a2/a9: X += sum of partials; A = RMSNorm(X) * gain.  final: also fp32 hidden.  A row is one block, as wide as
// blocks get: what bounds it is the chain of loads of a thread's columns.  (This and k_qkv_rope's second grid dimension:
// 1B-shaped fp32 cut of 4 layers, 10 rows, a step 763 -> 674 us on a B200.)
constexpr int kNormThreads = 1024;
template <typename T>
__global__ void __launch_bounds__(kNormThreads) k_reduce_norm(const StepArgs* __restrict__ args, Work w, Dims dm, SplitPlan sp, size_t slot_stride,
                              const T* __restrict__ gain, int final_norm) {
  extern __shared__ float xs[];
  __shared__ float red[32];
  pdl_wait();
  pdl_launch();
  const int r = blockIdx.x;
#pragma unroll 2
  for (int i = threadIdx.x; i < dm.d; i += blockDim.x) {
    float x = w.X[(size_t)r * dm.d + i] + reduce_partials(w.P, sp, slot_stride, dm.d, r, i);
    xs[i] = x;
    w.X[(size_t)r * dm.d + i] = x;
  }
  __syncthreads();
  float* hf = final_norm ? w.Hf + (size_t)r * dm.d : nullptr;
  float* dbg = (final_norm && args->dbg_hidden) ? args->dbg_hidden + (size_t)r * dm.d : nullptr;
  norm_row_from_smem<T>(xs, dm.d, gain, dm.eps, w.A, gridDim.x, r, hf, dbg, red);
}

// a9 of wide steps, whose last projection leaves the residual stream only: the final norm of every row.
template <typename T>
__global__ void k_final_norm(const StepArgs* __restrict__ args, Work w, Dims dm, const T* __restrict__ gain) {
  extern __shared__ float xs[];
  __shared__ float red[32];
  pdl_wait();
  pdl_launch();
  const int r = blockIdx.x;
  for (int i = threadIdx.x; i < dm.d; i += blockDim.x) xs[i] = w.X[(size_t)r * dm.d + i];
  __syncthreads();
  norm_row_from_smem<T>(xs, dm.d, gain, dm.eps, w.A, gridDim.x, r, w.Hf + (size_t)r * dm.d,
                        args->dbg_hidden ? args->dbg_hidden + (size_t)r * dm.d : nullptr, red);
}

// a3 tail + a4: reduce QKV partials, add bias, rotate q and k, store q, append k and v rows.  gridDim.y blocks share a row (with
// one block per row a thread walked through five pairs of dependent loads while most SMs had nothing to do).
template <typename T>
__global__ void k_qkv_rope(const StepArgs* __restrict__ args, KvView kv, Work w, Dims dm, SplitPlan sp,
                           size_t slot_stride, int layer, const T* __restrict__ bq, const T* __restrict__ bk,
                           const T* __restrict__ bv) {
  pdl_wait();
  pdl_launch();
  const int r = blockIdx.x, rows = args->gamma + 1;
  const int b = r / rows;
  const int seq = args->seq_ids[b];
  const int pos = w.row_pos[r];
  const int half = dm.hd / 2;
  const int qd = dm.Hq * dm.hd, kd = dm.Hkv * dm.hd, N = qd + 2 * kd;
  const bool store_kv = r < args->kv_rows;   // block-uniform
  const int page = store_kv ? kv.block_table[(size_t)seq * kv.max_pages_per_seq + pos / kv.page_size] : 0;
  const int slot = pos % kv.page_size;
  const float2* rt = w.rope + (size_t)r * half;
  // rotated heads: q heads then k heads
  const int first = blockIdx.y * blockDim.x + threadIdx.x, step = gridDim.y * blockDim.x;
  for (int p = first; p < (dm.Hq + dm.Hkv) * half; p += step) {
    int head = p / half, i = p % half;
    int n1 = head * dm.hd + i, n2 = n1 + half;
    float x1 = reduce_partials(w.P, sp, slot_stride, N, r, n1);
    float x2 = reduce_partials(w.P, sp, slot_stride, N, r, n2);
    if (head < dm.Hq) {
      if (bq) { x1 += to_f(bq[n1]); x2 += to_f(bq[n2]); }
    } else if (bk) {
      x1 += to_f(bk[n1 - qd]); x2 += to_f(bk[n2 - qd]);
    }
    float2 cs = rt[i];
    float y1 = x1 * cs.x - x2 * cs.y;
    float y2 = x2 * cs.x + x1 * cs.y;
    if (head < dm.Hq) {
      float* q = w.Q + (size_t)r * qd;
      q[n1] = y1;
      q[n2] = y2;
      if (w.Qb) {
        const int group = dm.Hq / dm.Hkv, j = r % rows;
        const float qs = 1.4426950408889634f / sqrtf((float)dm.hd);
        __half* qb = w.Qb + ((((size_t)b * dm.Hkv + head / group) * group + head % group) * rows + j) * dm.hd;
        const __half h1 = __float2half_rn(y1 * qs), h2 = __float2half_rn(y2 * qs);
        qb[i] = h1;
        qb[i + half] = h2;
        __half* ql = w.Qlo + (qb - w.Qb);
        ql[i] = __float2half_rn(y1 * qs - __half2float(h1));
        ql[i + half] = __float2half_rn(y2 * qs - __half2float(h2));
      }
    } else {
      if (store_kv) {
        T* krow = kv_row<T>(kv, layer, page, 0, head - dm.Hq, slot);
        krow[i] = from_f<T>(y1);
        krow[i + half] = from_f<T>(y2);
      }
      if (w.KVn) {
        __half* kn = w.KVn + ((((size_t)b * dm.Hkv + head - dm.Hq) * 2) * rows + r % rows) * dm.hd;
        kn[i] = __float2half_rn(y1);
        kn[i + half] = __float2half_rn(y2);
      }
    }
  }
  for (int p = first; p < kd; p += step) {
    float x = reduce_partials(w.P, sp, slot_stride, N, r, qd + kd + p);
    if (bv) x += to_f(bv[p]);
    if (store_kv) kv_row<T>(kv, layer, page, 1, p / dm.hd, slot)[p % dm.hd] = from_f<T>(x);
    if (w.KVn) w.KVn[((((size_t)b * dm.Hkv + p / dm.hd) * 2 + 1) * rows + r % rows) * dm.hd + p % dm.hd] = __float2half_rn(x);
  }
}

// a7 tail: H = silu(gate) * up from the partials of the fused [gate; up] projection.
template <typename T>
__global__ void k_swiglu(Work w, Dims dm, SplitPlan sp, size_t slot_stride) {
  pdl_wait();
  pdl_launch();
  const int r = blockIdx.y;
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= dm.F) return;
  float g = reduce_partials(w.P, sp, slot_stride, 2 * dm.F, r, f);
  float u = reduce_partials(w.P, sp, slot_stride, 2 * dm.F, r, dm.F + f);
  float y = g / (1.0f + expf(-g)) * u;
  store_act<T>(w.H, gridDim.y, dm.F, r, f, y);
}

// ---------------------------------------------------------------------------------------------
// CUDA-core skinny GEMM: a warp computes NF output features for RT rows, lanes over K.  Used for fp32 models
// and as a cross-check of the tensor-core kernel.
//
// What bounds it is the load path: every weight is used once per row, and its activations come from L1 / L2.  With one
// feature per warp a 16-byte weight load came with RT activation loads and the rows beyond RT = 8 read the weights again
// (1B-shaped fp32 model, 10 rows: 730 GB/s of weights, the GEMMs 2.8 ms of a 3.3 ms step).  NF = 4 features share each
// activation load, RT is picked to cover the rows in one pass where it can, and where N leaves SMs without a block, `ks`
// of a block's eight warps share a group of features and split K (their sums meet in shared memory, in warp order).
// ---------------------------------------------------------------------------------------------
struct GemmSegs {
  const void* w[3];  // up to three weight matrices stacked along the output dimension
  int rows[3];
  int nseg;
};

template <typename T> struct Vec;
template <> struct Vec<float> { typedef float4 type; static constexpr int n = 4; };
template <> struct Vec<bf16> { typedef uint4 type; static constexpr int n = 8; };

__device__ __forceinline__ void unpack(const float4& v, float* f) { f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w; }
__device__ __forceinline__ void unpack(const uint4& v, float* f) {
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float2 t = __bfloat1622float2(h[i]);
    f[2 * i] = t.x;
    f[2 * i + 1] = t.y;
  }
}

// Projections on the CUDA cores where k_gemm_f32 does not go: bf16 models without tensor-core options, and sj_gemm_skinny.
// `planes` = 2: the input is a hi/lo pair of bf16 planes (see Work); the two are added before use.
template <typename T, int RT, int NF>
__global__ void __launch_bounds__(256)
k_gemm_simt(const T* __restrict__ A, GemmSegs segs, float* __restrict__ Y, int R, int N, int K, int planes, int ks) {
  pdl_wait();
  pdl_launch();
  constexpr int VN = Vec<T>::n;
  typedef typename Vec<T>::type V;
  static_assert(NF * RT % 16 == 0, "sums are reduced sixteen at a time");
  __shared__ float part[8][NF * RT];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, kp = warp % ks;
  const int n0 = (blockIdx.x * (8 / ks) + warp / ks) * NF;   // past N in the last block's last warps: nothing is stored
  const T* wrow[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    int nn = min(n0 + f, N - 1), s = 0;   // features past the last repeat it and are not stored
    while (s < segs.nseg - 1 && nn >= segs.rows[s]) { nn -= segs.rows[s]; ++s; }
    wrow[f] = reinterpret_cast<const T*>(segs.w[s]) + (size_t)nn * K;
  }
#pragma unroll 1
  for (int r0 = 0; r0 < R; r0 += RT) {
    const T* arow[RT];   // rows past the last repeat it
#pragma unroll
    for (int i = 0; i < RT; ++i) arow[i] = A + (size_t)min(r0 + i, R - 1) * K;
    float acc[NF][RT];
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
      for (int i = 0; i < RT; ++i) acc[f][i] = 0.f;
    V wn[NF];   // the next step's weights, requested a step ahead
#pragma unroll
    for (int f = 0; f < NF; ++f) wn[f] = *reinterpret_cast<const V*>(wrow[f] + min((lane + 32 * kp) * VN, K - VN));
#pragma unroll 1
    for (int k = (lane + 32 * kp) * VN; k < K; k += 32 * VN * ks) {
      float wf[NF][VN];
#pragma unroll
      for (int f = 0; f < NF; ++f) unpack(wn[f], wf[f]);
      const int kn = min(k + 32 * VN * ks, K - VN);
#pragma unroll
      for (int f = 0; f < NF; ++f) wn[f] = *reinterpret_cast<const V*>(wrow[f] + kn);
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        float af[VN];
        unpack(*reinterpret_cast<const V*>(arow[i] + k), af);
        if (planes == 2) {
          float lo[VN];
          unpack(*reinterpret_cast<const V*>(arow[i] + (size_t)pad16(R) * K + k), lo);
#pragma unroll
          for (int e = 0; e < VN; ++e) af[e] += lo[e];
        }
#pragma unroll
        for (int f = 0; f < NF; ++f)
#pragma unroll
          for (int e = 0; e < VN; ++e) acc[f][i] = fmaf(af[e], wf[f][e], acc[f][i]);
      }
    }
#pragma unroll
    for (int g = 0; g < NF * RT / 16; ++g) {
      const float t = warp_sum_n<16>(&acc[0][0] + 16 * g, lane);
      if ((lane & 1) == 0) part[warp][16 * g + (lane >> 1)] = t;
    }
    __syncthreads();
    if (kp == 0)
      for (int e = lane; e < NF * RT; e += 32) {
        const int f = e / RT, i = e % RT;
        float v = 0.f;
        for (int u = 0; u < ks; ++u) v += part[warp + u][e];
        if (r0 + i < R && n0 + f < N) Y[(size_t)(r0 + i) * N + n0 + f] = v;
      }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// a5: causal grouped-query attention over the paged cache, split along the keys.
// Work item = (chunk of chunk_len keys of one sequence, KV head); all query heads of the group and
// all gamma+1 rows share the item's K/V.  Each item writes unnormalised partials (m, l, o).
//
// What bounds it at the caches it meets (a few hundred to a few thousand keys) is the length of an item's chain: find the
// item, its pages, its keys; scores; softmax; output.  So a chunk is one tile of 64 keys as a rule, a tile's loads are all
// in flight together and, where no row of this step is among its keys, requested before the wait for the previous kernel;
// scores and outputs are blocked in registers (a thread: one key x 6 queries, then one dimension x 6 queries), operands
// 16 bytes at a time.  1B-shaped cut of 4 layers, 2 sequences of 512 keys, 10 rows: a step 898 -> 763 us (B200).
// ---------------------------------------------------------------------------------------------
constexpr int kAttKT = 64;      // keys per inner tile
constexpr int kAttMaxQ = 96;    // query vectors per item: (Hq/Hkv) * (gamma+1)
constexpr int kAttThreads = 256;
constexpr int kAttQB = 6;       // queries blocked in registers
__host__ __device__ __forceinline__ size_t att_simt_smem(int nq, int hd) {   // queries, keys, values, scores, (m, l, alpha)
  return sizeof(float) * ((size_t)nq * hd + kAttKT * (hd + 4) + kAttKT * hd + (size_t)nq * kAttKT + 3 * nq);
}

__device__ __forceinline__ int find_seq(const int* chunk_start, int B, int chunk) {
  int lo = 0, hi = B - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (chunk_start[mid] <= chunk) lo = mid; else hi = mid - 1;
  }
  return lo;
}

template <typename T, int hd>
__global__ void __launch_bounds__(kAttThreads, hd == 64 ? 2 : 1)
k_attn_simt(const StepArgs* __restrict__ args, KvView kv, Work w, Dims dm, int layer, int chunk_len) {
  extern __shared__ __align__(16) float sm[];
  // The row positions, the chunk list and the cached rows are the work of kernels before the one that this one waits for.
  const int B = args->B, rows = args->gamma + 1;
  const int group = dm.Hq / dm.Hkv, nq = group * rows;
  float* qs = sm;                         // [nq][hd]
  float* ks = qs + nq * hd;               // [KT][hd + 4]
  float* vs = ks + kAttKT * (hd + 4);     // [KT][hd]
  float* ss = vs + kAttKT * hd;           // [nq][KT]
  float* m_run = ss + nq * kAttKT;        // [nq]
  float* l_run = m_run + nq;              // [nq]
  float* alpha = l_run + nq;              // [nq]
  const float scale = 1.0f / sqrtf((float)hd);
  const int total = w.chunk_start[B] * dm.Hkv;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int ng = kAttThreads / hd, NA = kAttMaxQ / ng;   // output: thread = dimension, ng groups of queries
  bool waited = false;

  for (int item = blockIdx.x; item < total; item += gridDim.x) {
    const int chunk = item / dm.Hkv, kvh = item % dm.Hkv;
    const int b = find_seq(w.chunk_start, B, chunk);
    const int seq = args->seq_ids[b];
    const int L = w.row_pos[b * rows];  // cached tokens before the block
    const int k_begin = (chunk - w.chunk_start[b]) * chunk_len;
    const int k_end = min(k_begin + chunk_len, L + rows);
    float acc[NA];   // queries grp + ng * i of this thread's dimension
#pragma unroll
    for (int i = 0; i < NA; ++i) acc[i] = 0.f;
    for (int k0 = k_begin; k0 < k_end; k0 += kAttKT) {
      constexpr int VN = Vec<T>::n, MAXV = kAttKT * hd / VN / kAttThreads;
      typedef typename Vec<T>::type V;
      V kv4[MAXV], vv4[MAXV];
      if (!waited && k0 + kAttKT > L) { pdl_wait(); pdl_launch(); waited = true; }   // rows of this step are among the keys
#pragma unroll
      for (int u = 0; u < MAXV; ++u) {
        const int i = (tid + u * kAttThreads) * VN, kk = i / hd, dd = i % hd, key = min(k0 + kk, k_end - 1);
        const int page = kv.block_table[(size_t)seq * kv.max_pages_per_seq + key / kv.page_size];
        const T* kr = kv_row<T>(kv, layer, page, 0, kvh, key % kv.page_size) + dd;
        kv4[u] = *reinterpret_cast<const V*>(kr);
        vv4[u] = *reinterpret_cast<const V*>(kr + (size_t)kv.n_kv_heads * kv.page_size * kv.head_dim);
      }
      if (!waited) { pdl_wait(); pdl_launch(); waited = true; }
      __syncthreads();   // the tile before has been read
      if (k0 == k_begin) {   // queries of this KV head's group: q index = g * rows + j
        for (int i = 4 * tid; i < nq * hd; i += 4 * kAttThreads) {
          const int q = i / hd, dd = i % hd, g = q / rows, j = q % rows;
          *reinterpret_cast<float4*>(qs + i) = *reinterpret_cast<const float4*>(w.Q + (size_t)(b * rows + j) * (dm.Hq * hd) + (kvh * group + g) * hd + dd);
        }
        for (int q = tid; q < nq; q += kAttThreads) { m_run[q] = -INFINITY; l_run[q] = 0.f; }
      }
#pragma unroll
      for (int u = 0; u < MAXV; ++u) {
        const int i = (tid + u * kAttThreads) * VN, kk = i / hd, dd = i % hd;
        float kf[VN], vf[VN];
        unpack(kv4[u], kf);
        unpack(vv4[u], vf);
        const bool live = k0 + kk < k_end;
#pragma unroll
        for (int e = 0; e < VN; e += 4) {
          *reinterpret_cast<float4*>(ks + kk * (hd + 4) + dd + e) = live ? make_float4(kf[e], kf[e + 1], kf[e + 2], kf[e + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
          *reinterpret_cast<float4*>(vs + kk * hd + dd + e) = live ? make_float4(vf[e], vf[e + 1], vf[e + 2], vf[e + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
      __syncthreads();
      // scores: thread = key, four groups of threads take queries tid / 64, + 4, ...
      {
        const int kk = tid & (kAttKT - 1), key = k0 + kk, q_first = tid / kAttKT;
        const float4* kr = reinterpret_cast<const float4*>(ks + kk * (hd + 4));
        constexpr int QS = kAttThreads / kAttKT;
        for (int q0 = q_first; q0 < nq; q0 += QS * kAttQB) {
          float a[kAttQB];
#pragma unroll
          for (int i = 0; i < kAttQB; ++i) a[i] = 0.f;
#pragma unroll 4
          for (int d4 = 0; d4 < hd / 4; ++d4) {
            const float4 kx = kr[d4];
#pragma unroll
            for (int i = 0; i < kAttQB; ++i) {
              const float4 qx = *reinterpret_cast<const float4*>(qs + min(q0 + QS * i, nq - 1) * hd + 4 * d4);
              a[i] = fmaf(qx.w, kx.w, fmaf(qx.z, kx.z, fmaf(qx.y, kx.y, fmaf(qx.x, kx.x, a[i]))));
            }
          }
#pragma unroll
          for (int i = 0; i < kAttQB; ++i) {
            const int q = q0 + QS * i;
            if (q < nq) ss[q * kAttKT + kk] = key < k_end && key <= L + q % rows ? a[i] * scale : -INFINITY;
          }
        }
      }
      __syncthreads();
      // online softmax: a warp per query, three side by side, two keys a lane
      constexpr int NW = kAttThreads / 32, SQ = 3;
      for (int q0 = warp; q0 < nq; q0 += NW * SQ) {
        float s0[SQ], s1[SQ], mx[SQ], sum[SQ], mo[SQ];
#pragma unroll
        for (int i = 0; i < SQ; ++i) {
          const int q = min(q0 + NW * i, nq - 1);
          s0[i] = ss[q * kAttKT + lane];
          s1[i] = ss[q * kAttKT + 32 + lane];
          mo[i] = m_run[q];
          mx[i] = fmaxf(s0[i], s1[i]);
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < SQ; ++i) mx[i] = fmaxf(mo[i], warp_max(mx[i]));
#pragma unroll
        for (int i = 0; i < SQ; ++i) {
          s0[i] = s0[i] == -INFINITY ? 0.f : expf(s0[i] - mx[i]);
          s1[i] = s1[i] == -INFINITY ? 0.f : expf(s1[i] - mx[i]);
          sum[i] = warp_sum(s0[i] + s1[i]);
        }
#pragma unroll
        for (int i = 0; i < SQ; ++i) {
          const int q = q0 + NW * i;
          if (q < nq) {   // warp-uniform
            ss[q * kAttKT + lane] = s0[i];
            ss[q * kAttKT + 32 + lane] = s1[i];
            if (lane == 0) {
              const float f = mx[i] == -INFINITY ? 1.f : (mo[i] == -INFINITY ? 0.f : expf(mo[i] - mx[i]));
              alpha[q] = f;
              l_run[q] = l_run[q] * f + sum[i];
              m_run[q] = mx[i];
            }
          }
        }
      }
      __syncthreads();
      // o[q][dd] = o * alpha + sum_k p[q][k] v[k][dd]
      const int dd = tid % hd, grp = tid / hd;
#pragma unroll
      for (int i0 = 0; i0 < NA; i0 += kAttQB)
        if (i0 * ng < nq) {   // block-uniform
          float a[kAttQB];
          const float* pq[kAttQB];
#pragma unroll
          for (int i = 0; i < kAttQB; ++i) {
            const int q = min(grp + ng * (i0 + i), nq - 1);
            pq[i] = ss + q * kAttKT;
            a[i] = acc[i0 + i] * alpha[q];
          }
#pragma unroll 4
          for (int kk = 0; kk < kAttKT; kk += 4) {
            const float v0 = vs[kk * hd + dd], v1 = vs[(kk + 1) * hd + dd], v2 = vs[(kk + 2) * hd + dd], v3 = vs[(kk + 3) * hd + dd];
#pragma unroll
            for (int i = 0; i < kAttQB; ++i) {
              const float4 p = *reinterpret_cast<const float4*>(pq[i] + kk);
              a[i] = fmaf(p.w, v3, fmaf(p.z, v2, fmaf(p.y, v1, fmaf(p.x, v0, a[i]))));
            }
          }
#pragma unroll
          for (int i = 0; i < kAttQB; ++i) acc[i0 + i] = a[i];
        }
    }
    __syncthreads();
    // partials: index ((chunk * Hq + head) * rows + j)
    const size_t p0 = ((size_t)chunk * dm.Hq + kvh * group) * rows;   // query q of the group is p0 + q
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int q = tid / hd + ng * i;
      if (q < nq) w.att_o[(p0 + q) * hd + tid % hd] = acc[i];
    }
    for (int q = tid; q < nq; q += kAttThreads) {
      w.att_m[p0 + q] = m_run[q];
      w.att_l[p0 + q] = l_run[q];
    }
  }
  if (!waited) { pdl_wait(); pdl_launch(); }
}

// Merge the partials of one (row, head) over its sequence's chunks, in chunk order: a warp each, the chunks' maxima and sums
// one per lane, four chunks' outputs in flight.
constexpr int kSimtMergeThreads = 128;
template <typename T>
__global__ void __launch_bounds__(kSimtMergeThreads) k_attn_combine(const StepArgs* __restrict__ args, Work w, Dims dm, int R) {
  const int rows = args->gamma + 1, lane = threadIdx.x & 31;
  const int item = blockIdx.x * (kSimtMergeThreads / 32) + (threadIdx.x >> 5), r = item / dm.Hq, h = item % dm.Hq;
  const int b = min(r, R - 1) / rows, j = r % rows;
  const int c0 = w.chunk_start[b], c1 = w.chunk_start[b + 1];   // written before the kernel that this one waits for
  pdl_wait();
  pdl_launch();
  if (r >= R) return;
  const int n = c1 - c0, dpl = dm.hd / 32;   // 2 or 4 dimensions per lane
  const size_t p0 = ((size_t)c0 * dm.Hq + h) * rows + j, step = (size_t)dm.Hq * rows;
  const float2* o2 = reinterpret_cast<const float2*>(w.att_o + p0 * dm.hd) + lane;
  const size_t step2 = step * dm.hd / 2;
  float M = -INFINITY, lsum = 0.f;
  float2 o[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  for (int k0 = 0; k0 < n; k0 += 32) {
    const int kn = min(32, n - k0);
    const bool live = lane < kn;
    const float m = live ? __ldcg(w.att_m + p0 + (size_t)(k0 + lane) * step) : -INFINITY, l = live ? __ldcg(w.att_l + p0 + (size_t)(k0 + lane) * step) : 0.f;
    const float Mn = fmaxf(M, warp_max(m)), f = M == -INFINITY ? 0.f : expf(M - Mn);
    const float wt = m == -INFINITY ? 0.f : expf(m - Mn);
    lsum = lsum * f + warp_sum(l * wt);
    M = Mn;
#pragma unroll
    for (int e = 0; e < 2; ++e) { o[e].x *= f; o[e].y *= f; }
    for (int k = 0; k < kn; k += 4) {
      float2 x[4][2];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int e = 0; e < 2; ++e)
          if (2 * e < dpl) x[u][e] = __ldcg(o2 + (size_t)(k0 + min(k + u, kn - 1)) * step2 + 32 * e);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float wu = __shfl_sync(0xffffffffu, wt, min(k + u, 31));
#pragma unroll
        for (int e = 0; e < 2; ++e)
          if (2 * e < dpl && k + u < kn) { o[e].x += x[u][e].x * wu; o[e].y += x[u][e].y * wu; }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < 2; ++e)
    if (2 * e < dpl) {
      store_act<T>(w.ATT, R, dm.Hq * dm.hd, r, h * dm.hd + 64 * e + 2 * lane, o[e].x / lsum);
      store_act<T>(w.ATT, R, dm.Hq * dm.hd, r, h * dm.hd + 64 * e + 2 * lane + 1, o[e].y / lsum);
    }
}

// Dot product of GEMM-input row r (both bf16 planes) with one weight row, over the whole warp.
__device__ __forceinline__ float planes_dot(const bf16* __restrict__ A, int R, int K, int r, const bf16* __restrict__ wrow,
                                            int lane) {
  const bf16* hi = A + (size_t)r * K;
  const bf16* lo = A + ((size_t)pad16(R) + r) * K;
  float acc = 0.f;
  for (int k = lane; k < K; k += 32) acc = fmaf(__bfloat162float(hi[k]) + __bfloat162float(lo[k]), __bfloat162float(wrow[k]), acc);
  return warp_sum(acc);
}

// Top-k alignment test with the tensor-core LM head, which stores no logits: the logit of row j's drafted token
// d_{j+1} is computed ahead of the LM head (one dot product per row), so that the head's epilogue can count, tile
// by tile, how many logits rank before it.  One warp per row; idle unless the step asks for top_k >= 2.
static __global__ void k_target_logits(const StepArgs* __restrict__ args, Work w, Dims dm, const bf16* __restrict__ lm_head, int R) {
  pdl_wait();
  pdl_launch();
  if (args->top_k < 2) return;
  const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= R) return;
  const int rows = args->gamma + 1, b = r / rows, j = r % rows;
  if (j >= args->gamma) return;
  const int tok = min(max(args->draft_ids[b * args->gamma + j], 0), dm.V - 1);
  const float z = planes_dot(reinterpret_cast<const bf16*>(w.A), R, dm.d, r, lm_head + (size_t)tok * dm.d, lane);
  if (lane == 0) w.tgt_pre[r] = z;
}

// ---------------------------------------------------------------------------------------------
// a10 (CUDA-core path): per-(128-token vocabulary tile, row) softmax statistics from stored logits
// ---------------------------------------------------------------------------------------------
static __global__ void k_lm_stats_from_logits(const StepArgs* __restrict__ args, Work w, Dims dm, int R) {
  pdl_wait();
  pdl_launch();
  const int tile = blockIdx.x, lane = threadIdx.x & 31;
  const int r = blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (r >= R) return;
  const int rows = args->gamma + 1, b = r / rows, j = r % rows;
  const float invT = args->inv_temperature;
  const float* lg = w.logits + (size_t)r * dm.V;
  const int tgt = (j < args->gamma) ? args->draft_ids[b * args->gamma + j] : -1;
  float z[4];
  float m = -INFINITY;
  int arg = 0x7fffffff;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int v = tile * kTileN + i * 32 + lane;
    float raw = (v < dm.V) ? lg[v] : -INFINITY;
    if (v < dm.V && args->dbg_logits) args->dbg_logits[(size_t)r * dm.V + v] = raw;
    z[i] = raw * invT;
    if (v == tgt) w.tgt_logit[r] = z[i];
    if (z[i] > m) { m = z[i]; arg = v; }   // increasing v: strict > keeps the lowest index
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    float om = __shfl_xor_sync(0xffffffffu, m, o);
    int oa = __shfl_xor_sync(0xffffffffu, arg, o);
    if (om > m || (om == m && oa < arg)) { m = om; arg = oa; }
  }
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) s += (z[i] == -INFINITY) ? 0.f : expf(z[i] - m);
  s = warp_sum(s);
  int before = 0;   // top-k test: this tile's logits that rank before the drafted token's (the logits are stored here)
  if (args->top_k >= 2 && tgt >= 0) {
    const float zd = lg[min(tgt, dm.V - 1)];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int v = tile * kTileN + i * 32 + lane;
      const float raw = (v < dm.V) ? lg[v] : -INFINITY;
      const bool bf = v < dm.V && v != tgt && (raw > zd || (raw == zd && v < tgt));
      before += __popc(__ballot_sync(0xffffffffu, bf));
    }
  }
  if (lane == 0) {
    RowStat st; st.m = m; st.s = s; st.arg = arg; st.pad = before;
    w.stats[(size_t)tile * R + r] = st;
  }
}

// ---------------------------------------------------------------------------------------------
// a10 tail + a11..a15: merge statistics, judge scores, acceptance bits, first rejection, next
// token (greedy), new cache length and commit.  One block per sequence.
// ---------------------------------------------------------------------------------------------
static __global__ void k_finalize(const StepArgs* __restrict__ args, KvView kv, Work w, Dims dm, int n_vtiles, int R) {
  pdl_wait();
  pdl_launch();
  __shared__ RowStat part[kMaxGamma + 1][2];
  __shared__ RowStat rs[kMaxGamma + 1];
  __shared__ float score[kMaxGamma + 1];
  const int b = blockIdx.x, gamma = args->gamma, rows = gamma + 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  const int seq = args->seq_ids[b];
  merge_row_stats(w.stats, n_vtiles, R, b * rows, rows, warp, lane, part);
  // judge scores: Verifier(h_j) = sigmoid(w.h_j + b), j = 1..gamma, one warp per row
  for (int j = 1 + warp; j <= gamma; j += nwarp) {
    const float* h = w.Hf + (size_t)(b * rows + j) * dm.d;
    float a = 0.f;
    if (args->has_judge) {
#pragma unroll 8
      for (int i = 4 * lane; i < dm.d; i += 128) {   // d is a multiple of 8
        const float4 hv = *reinterpret_cast<const float4*>(h + i), jv = *reinterpret_cast<const float4*>(w.judge_w + i);
        a = fmaf(hv.x, jv.x, fmaf(hv.y, jv.y, fmaf(hv.z, jv.z, fmaf(hv.w, jv.w, a))));
      }
    }
    a = warp_sum(a);
    if (lane == 0) {
      float s = args->has_judge ? 1.0f / (1.0f + expf(-(a + args->judge_bias))) : 0.f;
      score[j] = s;
      args->judge_scores[b * gamma + j - 1] = s;
    }
  }
  __syncthreads();
  if (tid < rows) {
    rs[tid] = merge_row_halves(part[tid]);
    w.rowstat[b * rows + tid] = rs[tid];
  }
  __syncthreads();
  if (warp == 0) {
    bool ok = true;  // lanes >= gamma do not constrain the scan
    if (lane < gamma) {
      const int j = lane + 1;  // drafted position
      const int d = args->draft_ids[b * gamma + lane];
      const RowStat st = rs[j - 1];
      const float zd = w.tgt_logit[b * rows + j - 1] - st.m;
      const float p = expf(zd) / st.s;
      args->p_draft[b * gamma + lane] = p;
      if (args->logp_draft) args->logp_draft[b * gamma + lane] = zd - logf(st.s);
      bool align;
      if (args->mode == 0) align = args->top_k >= 2 ? st.pad < args->top_k : (d == st.arg);
      else align = args->uniforms[b * rows + lane] * args->q_tok[b * gamma + lane] < p;
      bool judge = args->has_judge && (score[j] > args->theta[b]);
      ok = (args->use_align && align) || (args->use_judge && judge) || args->accept_all;
    }
    unsigned rej = __ballot_sync(0xffffffffu, !ok);
    int n = rej ? (__ffs(rej) - 1) : gamma;
    if (lane == 0) {
      const int L = w.row_pos[b * rows];
      args->accepted_len[b] = n;
      args->new_kv_len[b] = L + 1 + n;
      if (args->mode == 0) {
        int nxt = rs[n].arg;
        args->next_token[b] = nxt;
        if (args->commit) kv.pending[seq] = nxt;
      }
      if (args->commit) kv.kv_len[seq] = L + 1 + n;
    }
  }
}

// One row of the residual stream (the last of a prefill) through the final norm into GEMM input planes of their own.
template <typename T>
__global__ void k_select_row(Work w, Dims dm, const T* __restrict__ gain, int row) {
  extern __shared__ float xs[];
  __shared__ float red[32];
  pdl_wait();
  pdl_launch();
  for (int i = threadIdx.x; i < dm.d; i += blockDim.x) xs[i] = w.X[(size_t)row * dm.d + i];
  __syncthreads();
  norm_row_from_smem<T>(xs, dm.d, gain, dm.eps, w.Asel, 1, 0, nullptr, nullptr, red);
}

// a14, sampling mode: inverse CDF over the vocabulary of norm(max(0, p_n - q_{n+1})) (first
// rejection) or of p_gamma (everything accepted), driven by uniforms[:, gamma].  fp64 prefix sums.
//
// The LM head's pass has stored the logits of all rows (4 bytes an entry against the 2 d bytes of weights that a second
// pass over the chosen row would read).  One block of 1024 threads per sequence that walked the row in 1024 contiguous
// pieces spent its time on a chain of uncoalesced loads and fp64 adds; now chunks of kResampleChunk entries are summed by a
// block each, and one block per sequence finds the chunk and the entry.  The second pass and the old draw took 350 us of a
// step of an 8B-shaped target (128256 entries), what is left of both 20 (B200).
constexpr int kResampleThreads = 256, kResamplePer = 8, kResampleChunk = kResampleThreads * kResamplePer;

struct ResampleRow {
  const float* lg;   // the row's logits
  const float* q;    // the draft's probabilities there; null: everything was accepted
  float invT, m;
  double inv_s;
};
__device__ __forceinline__ ResampleRow resample_row(const StepArgs* args, const Work& w, const Dims& dm, int b) {
  const int gamma = args->gamma, n = args->accepted_len[b], r = b * (gamma + 1) + n;
  const RowStat st = w.rowstat[r];
  return ResampleRow{w.logits + (size_t)r * dm.V, n < gamma ? args->q_full + ((size_t)b * gamma + n) * dm.V : nullptr,
                     args->inv_temperature, st.m, 1.0 / (double)st.s};
}
// This thread's kResamplePer entries of chunk c: p, and max(0, p - q) in `res`; 0 beyond the vocabulary.
__device__ __forceinline__ void resample_load(const ResampleRow& x, int V, int c, double (&p)[kResamplePer], double (&res)[kResamplePer]) {
  const int v0 = c * kResampleChunk + (int)threadIdx.x * kResamplePer;
  float lg[kResamplePer], q[kResamplePer];
#pragma unroll
  for (int i = 0; i < kResamplePer; ++i) {
    lg[i] = __ldcg(x.lg + min(v0 + i, V - 1));
    q[i] = x.q ? x.q[min(v0 + i, V - 1)] : 0.f;
  }
#pragma unroll
  for (int i = 0; i < kResamplePer; ++i) {
    p[i] = v0 + i < V ? (double)expf(lg[i] * x.invT - x.m) * x.inv_s : 0.0;
    res[i] = fmax(0.0, p[i] - (double)q[i]);
  }
}
// Inclusive prefix sum over the block's threads, left in sm[1 ..]; sm[0] = 0.  sm: [kResampleThreads + 1 + 8].
__device__ __forceinline__ void resample_scan(double v, double* sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const double up = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += up;
  }
  double* wsum = sm + kResampleThreads + 1;
  if (lane == 31) wsum[warp] = v;
  __syncthreads();
  double before = 0.0;
  for (int k = 0; k < warp; ++k) before += wsum[k];
  sm[threadIdx.x + 1] = before + v;
  if (threadIdx.x == 0) sm[0] = 0.0;
  __syncthreads();
}

// grid (chunks, B): the chunk's sums of p and of max(0, p - q)
static __global__ void k_resample_sums(const StepArgs* __restrict__ args, Work w, Dims dm) {
  pdl_wait();
  pdl_launch();
  __shared__ double sm[kResampleThreads + 9];
  const int c = blockIdx.x, b = blockIdx.y;
  double p[kResamplePer], res[kResamplePer], tp = 0.0, tr = 0.0;
  resample_load(resample_row(args, w, dm, b), dm.V, c, p, res);
#pragma unroll
  for (int i = 0; i < kResamplePer; ++i) { tp += p[i]; tr += res[i]; }
  double2 out;
  resample_scan(tp, sm);
  out.x = sm[kResampleThreads];
  __syncthreads();
  resample_scan(tr, sm);
  out.y = sm[kResampleThreads];
  if (threadIdx.x == 0) w.rs_part[(size_t)b * gridDim.x + c] = out;
}

// grid B: the chunk, then the entry, whose prefix sum first exceeds u times the total
static __global__ void k_resample_pick(const StepArgs* __restrict__ args, KvView kv, Work w, Dims dm, int n_chunks) {
  pdl_wait();
  pdl_launch();
  __shared__ double sm[kResampleThreads + 9];
  __shared__ int pick, last;
  const int b = blockIdx.x, tid = threadIdx.x, rows = args->gamma + 1;
  const ResampleRow x = resample_row(args, w, dm, b);
  const double2* part = w.rs_part + (size_t)b * n_chunks;
  double total_p = 0.0, total_r = 0.0;
  for (int c0 = 0; c0 < n_chunks; c0 += kResampleThreads) {
    const double2 v = c0 + tid < n_chunks ? __ldcg(part + c0 + tid) : make_double2(0.0, 0.0);
    resample_scan(v.x, sm);
    total_p += sm[kResampleThreads];
    __syncthreads();
    resample_scan(v.y, sm);
    total_r += sm[kResampleThreads];
    __syncthreads();
  }
  const bool residual = x.q != nullptr && total_r > 0.0;   // no residual mass: fall back to p
  const double target = (double)args->uniforms[b * rows + args->gamma] * (residual ? total_r : total_p);
  double carry = 0.0;
  int chunk = -1;
  for (int c0 = 0; c0 < n_chunks && chunk < 0; c0 += kResampleThreads) {
    if (tid == 0) pick = kResampleThreads;
    const double2 v = c0 + tid < n_chunks ? __ldcg(part + c0 + tid) : make_double2(0.0, 0.0);
    resample_scan(residual ? v.y : v.x, sm);
    if (carry + sm[tid + 1] > target) atomicMin(&pick, tid);
    __syncthreads();
    const int k = pick;
    if (k < kResampleThreads) {
      chunk = c0 + k;
      carry += sm[k];
    } else {
      carry += sm[kResampleThreads];
    }
    __syncthreads();
  }
  if (tid == 0) { pick = kResampleThreads; last = -1; }
  double p[kResamplePer], res[kResamplePer], own = 0.0;
  if (chunk >= 0) {
    resample_load(x, dm.V, chunk, p, res);
#pragma unroll
    for (int i = 0; i < kResamplePer; ++i) {
      if (residual) p[i] = res[i];
      own += p[i];
    }
  }
  resample_scan(own, sm);
  if (carry + sm[tid + 1] > target) atomicMin(&pick, tid);
  if (own > 0.0) atomicMax(&last, tid);   // a sum that rounding left short of the target ends at the last entry with mass
  __syncthreads();
  const int who = chunk < 0 ? 0 : (pick < kResampleThreads ? pick : max(last, 0));
  if (tid == who) {
    int winner = dm.V - 1;
    if (chunk >= 0) {
      const int v0 = chunk * kResampleChunk + tid * kResamplePer;
      double run = 0.0;
      bool found = false;
#pragma unroll
      for (int i = 0; i < kResamplePer; ++i) {
        run += p[i];
        if (!found && p[i] > 0.0) { winner = v0 + i; found = carry + (sm[tid] + run) > target; }
      }
    }
    args->next_token[b] = winner;
    if (args->commit) kv.pending[args->seq_ids[b]] = winner;
  }
}

// The end of a prefill block of n tokens: the sequence is n tokens longer; with `stats` (softmax statistics of the last
// token's row per vocabulary tile) its arg max becomes the pending token.
static __global__ void k_prefill_commit(KvView kv, int seq, int n, const RowStat* __restrict__ stats, int n_vtiles, int* next) {
  pdl_wait();
  pdl_launch();
  __shared__ RowStat sred[256];
  const int tid = threadIdx.x;
  if (stats) {
    RowStat a; a.m = -INFINITY; a.s = 0.f; a.arg = 0; a.pad = 0;
    const int per = (n_vtiles + 255) / 256, t1 = min((tid + 1) * per, n_vtiles);
    for (int t = tid * per; t < t1; ++t) a = stat_merge(a, stats[t]);
    sred[tid] = a;
    __syncthreads();
    for (int stride = 1; stride < 256; stride <<= 1) {
      if ((tid & (2 * stride - 1)) == 0) sred[tid] = stat_merge(sred[tid], sred[tid + stride]);
      __syncthreads();
    }
  }
  if (tid == 0) {
    if (stats) {
      *next = sred[0].arg;
      kv.pending[seq] = sred[0].arg;
    }
    kv.kv_len[seq] += n;
  }
}

// Rollback: kv_len <- new_len where new_len <= kv_len, else flag the error and leave it; a sequence named more than once ends at the
// shortest.  One thread per entry, one block.
static __global__ void __launch_bounds__(kMaxEdits) k_rollback(KvView kv, const __grid_constant__ KvEdits to, int* status) {
  const bool live = (int)threadIdx.x < to.n;
  const int s = to.e[live ? threadIdx.x : 0].seq, n = to.e[live ? threadIdx.x : 0].value;
  const bool ok = live && n >= 0 && n <= kv.kv_len[s];
  __syncthreads();   // every entry is held against the length before the call
  if (ok) atomicMin(&kv.kv_len[s], n);
  else if (live) atomicCAS(status, DEV_OK, DEV_STATE);
}

// Copy rows between a contiguous [n, Hkv, hd] buffer and the paged pool (fill: to_pool = 1).
template <typename T>
__global__ void k_kv_copy(KvView kv, int seq, int layer, int start, int n_tokens, T* k, T* v, int to_pool) {
  const int t = blockIdx.x;
  if (t >= n_tokens) return;
  const int pos = start + t;
  const int page = kv.block_table[(size_t)seq * kv.max_pages_per_seq + pos / kv.page_size];
  const int slot = pos % kv.page_size;
  const int width = kv.n_kv_heads * kv.head_dim;
  for (int i = threadIdx.x; i < width; i += blockDim.x) {
    int h = i / kv.head_dim, dd = i % kv.head_dim;
    T* kr = kv_row<T>(kv, layer, page, 0, h, slot) + dd;
    T* vr = kv_row<T>(kv, layer, page, 1, h, slot) + dd;
    if (to_pool) { *kr = k[(size_t)t * width + i]; *vr = v[(size_t)t * width + i]; }
    else { k[(size_t)t * width + i] = *kr; v[(size_t)t * width + i] = *vr; }
  }
}

}  // namespace sj
