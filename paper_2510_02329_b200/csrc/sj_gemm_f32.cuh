// Projections and LM head of fp32 models, on the CUDA cores (the tensor cores take no fp32 operands).
//
//   Y[slot][R, N] (fp32) = A[R, K] . W[N, K]^T
// A block computes tiles of 64 features for up to RT rows at a time: eight warps, each 8 features x RT rows, lanes over K.
// Weights and activations come through a ring in shared memory (cp.async, 16 bytes a thread) in steps of 128 of K.
//
// What bounds it is HBM, so the ring (five stages of 32 KiB of weights, one block per SM) keeps 160 KiB per SM on the way;
// a step's 32 RT FMAs and 8 + RT shared-memory loads a lane take about 900 of the 1400 clocks in which HBM delivers its
// weights at 12 rows.  Loading straight into registers a step ahead (k_gemm_simt) kept 32 KiB on the way and read each
// activation once per four features from L1.  Work is dealt in units (tile, K step), evenly to one block per SM, so that
// every SM streams the same bytes whatever N is; a tile that several blocks share leaves a slot of sums per block, added in
// block order by the kernel that reads them (SplitPlan).  1B-shaped cut of 4 layers, 2 sequences of 512 keys, 10 rows, one cache
// replayed back to back: a step 1159 -> 898 us (B200).
//
// Rows beyond RT take another pass over a block's share of the tile, at most 256 K bytes: from L2 where 148 shares fit it (K = 2048: 78
// MB), from HBM again where they do not (K above 3300 or so where a tile is one block's, as in the LM head).  A step of 200 keys with
// k_gemm_simt and the attention and row kernels of its time, and now: 1B-shaped, 4 layers, 12 rows 1239 -> 718 us, 24 rows 2439 -> 1180, 96 rows
// 8824 -> 4035; 8B-shaped, 2 layers (K 4096 and 14336), 12 rows 1659 -> 665, 24 rows 3199 -> 1148, 512 rows 66455 -> 21704.
#pragma once

#include "sj_kernels.cuh"

namespace sj {

constexpr int kF32Feats = 64, kF32Shift = 6, kF32K = 128, kF32Threads = 256, kF32Stages = 5;
__host__ __device__ __forceinline__ int f32_stage_floats(int rt) { return (kF32Feats + rt) * kF32K; }

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool live) {   // 16 bytes; zeros where not live
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(live ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Block c's units of U dealt to G blocks are [c U / G, (c + 1) U / G).  The block that holds unit u:
__host__ __device__ __forceinline__ int f32_owner(int u, int U, int G) { return (int)((((long long)u + 1) * G - 1) / U); }

// Walks a block's work: for each tile its run of K steps, once per pass over the rows.
struct F32Cursor {
  int tile, kc, pass, kc_lo, kc_hi, hi, KC, n_pass;
  __device__ __forceinline__ void start(int lo, int hi_, int KC_, int n_pass_) {
    hi = hi_; KC = KC_; n_pass = n_pass_;
    tile = lo / KC;
    pass = 0;
    kc = kc_lo = lo % KC;
    kc_hi = min(KC, hi - tile * KC);
  }
  __device__ __forceinline__ bool done() const { return tile * KC + kc_lo >= hi; }
  __device__ __forceinline__ void next() {
    if (++kc < kc_hi) return;
    kc = kc_lo;
    if (++pass < n_pass) return;
    pass = 0;
    ++tile;
    kc = kc_lo = 0;
    kc_hi = min(KC, hi - tile * KC);
  }
};

// units: K steps of all tiles, or (whole) tiles, dealt to gridDim.x blocks.  rows_pp: rows of a pass, at most RT.
template <int RT>
__global__ void __launch_bounds__(kF32Threads, 1)
k_gemm_f32(const float* __restrict__ A, GemmSegs segs, float* __restrict__ Y, size_t slot_stride, int R, int N, int K, int rows_pp, int whole) {
  static_assert(RT % 2 == 0, "a group of 16 sums is two rows of eight features");
  extern __shared__ __align__(16) float f32_ring[];
  pdl_launch();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = blockIdx.x, G = gridDim.x;
  const int KC = (K + kF32K - 1) / kF32K, n_tiles = (N + kF32Feats - 1) / kF32Feats, U = n_tiles * KC;
  const int lo = whole ? (int)((long long)c * n_tiles / G) * KC : (int)((long long)c * U / G);
  const int hi = whole ? (int)((long long)(c + 1) * n_tiles / G) * KC : (int)((long long)(c + 1) * U / G);
  const int n_pass = (R + rows_pp - 1) / rows_pp;
  constexpr int stage_floats = (kF32Feats + RT) * kF32K;

  // this warp's 8 features of a step (segments begin at multiples of 8; features past the last repeat it)
  const float* wbase = nullptr;
  int wrows = 0, wtile = -1, wn = 0;
  auto load_w = [&](const F32Cursor& x, int stage) {
    if (x.tile != wtile) {
      wtile = x.tile;
      wn = min(x.tile * kF32Feats + warp * 8, N - 1);
      int s = 0;
      while (s < segs.nseg - 1 && wn >= segs.rows[s]) { wn -= segs.rows[s]; ++s; }
      wbase = reinterpret_cast<const float*>(segs.w[s]);
      wrows = segs.rows[s];
    }
    const int k = x.kc * kF32K + 4 * lane;
    float* dst = f32_ring + stage * stage_floats + warp * 8 * kF32K + 4 * lane;
#pragma unroll
    for (int f = 0; f < 8; ++f) cp_async16(dst + f * kF32K, wbase + (size_t)min(wn + f, wrows - 1) * K + min(k, K - 4), k < K);
  };
  auto load_a = [&](const F32Cursor& x, int stage) {
    const int k = x.kc * kF32K + 4 * lane;
    float* dst = f32_ring + stage * stage_floats + kF32Feats * kF32K + 4 * lane;
#pragma unroll
    for (int r = 0; r < RT; r += 8)
      if (r + warp < RT) cp_async16(dst + (r + warp) * kF32K, A + (size_t)min(x.pass * rows_pp + r + warp, R - 1) * K + min(k, K - 4), k < K);
  };

  F32Cursor in, out;
  in.start(lo, hi, KC, n_pass);
  out = in;
  // the first steps' weights do not depend on the kernel before this one
  F32Cursor w0 = in;
#pragma unroll
  for (int s = 0; s < kF32Stages - 1; ++s)
    if (!w0.done()) { load_w(w0, s); w0.next(); }
  pdl_wait();
#pragma unroll
  for (int s = 0; s < kF32Stages - 1; ++s) {
    if (!in.done()) { load_a(in, s); in.next(); }
    cp_async_commit();
  }

  float acc[RT][8];
#pragma unroll
  for (int r = 0; r < RT; ++r)
#pragma unroll
    for (int f = 0; f < 8; ++f) acc[r][f] = 0.f;
  int stage = 0;
#pragma unroll 1
  while (!out.done()) {
    cp_async_wait<kF32Stages - 2>();
    __syncthreads();   // everybody's part of this step is here, and everybody is done with the step before
    {
      const int into = stage == 0 ? kF32Stages - 1 : stage - 1;
      if (!in.done()) { load_w(in, into); load_a(in, into); in.next(); }
      cp_async_commit();
    }
    const float* st = f32_ring + stage * stage_floats + 4 * lane;
    float4 w[8];
#pragma unroll
    for (int f = 0; f < 8; ++f) w[f] = *reinterpret_cast<const float4*>(st + (warp * 8 + f) * kF32K);
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      const float4 a = *reinterpret_cast<const float4*>(st + (kF32Feats + r) * kF32K);
#pragma unroll
      for (int f = 0; f < 8; ++f) acc[r][f] = fmaf(a.w, w[f].w, fmaf(a.z, w[f].z, fmaf(a.y, w[f].y, fmaf(a.x, w[f].x, acc[r][f]))));
    }
    if (++stage == kF32Stages) stage = 0;
    const int tile = out.tile, r0 = out.pass * rows_pp;
    const bool last = out.kc + 1 == out.kc_hi;
    out.next();
    if (!last) continue;
    // the run of this (tile, pass) is complete: sums over the lanes to the block's slot of the tile
    const int n0 = tile * kF32Feats + warp * 8, slot = whole ? 0 : c - f32_owner(tile * KC, U, G);
    float* y = Y + (size_t)slot * slot_stride;
#pragma unroll
    for (int r = 0; r < RT; r += 2) {   // sixteen sums at a time: two rows of eight features
      const float t = warp_sum_n<16>(&acc[r][0], lane);
      const int row = r + (lane >> 4), n = n0 + ((lane >> 1) & 7);
      if ((lane & 1) == 0 && row < rows_pp && r0 + row < R && n < N) y[(size_t)(r0 + row) * N + n] = t;
    }
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
      for (int f = 0; f < 8; ++f) acc[r][f] = 0.f;
  }
}

}  // namespace sj
