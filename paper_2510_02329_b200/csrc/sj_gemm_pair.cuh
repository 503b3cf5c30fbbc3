// Projections of the per-stage step on pairs of SMs, with fused epilogues.
//
//   D[256 features, rb rows] (fp32, tensor memory) = W_tile[256, K] (bf16) x A[rb, K]^T (two bf16 planes)
// A pair of CTAs (tcgen05 cta_group::2) computes one 256-feature tile for a block of rb <= 128 rows over the whole of K:
// CTA `rank` holds the weights and the accumulator of features [128 rank, +128).  The MMA's N = 2 rb columns are the
// block's rows twice: the hi plane, staged by rank 0, and the lo plane, staged by rank 1; each SM's tensor core reads
// both.  The epilogue adds the two halves.
//
// The tensor core's accumulation truncates (measured against fp64: a chain of 896 MMAs comes out 1.4e-5 too small, one
// of 64 about 1e-6), so K is summed in segments of up to kPairSegKB K blocks whose results the epilogue warps add in fp32
// registers.  Segments alternate between two accumulators: the adding, and an item's epilogue, run beside the next
// segment's MMAs.
//
// Why this shape: what bounds wide steps is the shared-memory port (128 B/clk per SM).  A K step of 64 writes
// 16 KiB of weights and 128 rb bytes of activations and its four MMAs read 4 (4096 + 32 rb) back: 256 + 2 rb clocks, for
// 4 rb clocks of tensor time (512 and 512 at rb = 128).  A single CTA with both planes of 288 rows needs 1790 clocks for
// 1152 of tensor time.  Cutting the rows instead of K costs re-reads of the weights from L2 (pairs that share a tile
// run side by side) but no exchange of sums: a first version of this kernel that split K over the pairs was bound by
// the pair that finished a tile for all of them.
//
// Where the items (tile, row block) leave pairs idle (down has 16 to 20 tiles of 256 features), a cluster of n_split <= 4
// pairs shares an item's K.  Every pair sends its sums of the rows that another one finishes into that one's shared
// memory and finishes its own: the rows [32 j, 32 j + 32) of a block belong to split j % n_split, so all of them work on the
// epilogue (split 0 does all of a block of 16 rows) and no sum crosses L2.  A cluster is scheduled as a whole, so its pairs can wait for one another.
// The sums go as st.async: their arrival is the signal.  (A release after plain stores is one more trip: 1B-shaped 48 rows
// 954 -> 934 us a step, 8B-shaped 44 rows 4459 -> 4377, with the residual rows requested beside the MMAs.)
// Down at 72 rows (20 tiles, K 27648, 283 MB): 94.5 us with row blocks of 32 on 60 pairs, 60.4 as 80 rows on 40 pairs;
// steps (B200): 32B-shaped 72 rows 5434 -> 4871 us, 8B-shaped 44 rows 5150 -> 4440, 1B-shaped 48 rows 1610 -> 1447.
//
// Items, row blocks fastest, are dealt round robin: cluster g takes items g, g + n_groups, ...  The host picks rb and
// n_split by the model above (pair_geom).
//
// Epilogues (template SITE) -- the same arithmetic as the persistent kernel's: the planes hold x * gain and the row scalar
// 1/rms, from per-tile sums of squares, is applied by the consumer.
//   QKV  -> 1/rms, bias, rotary embedding; queries (fp16), K / V rows into the pages (bf16) and the step's side buffer
//   O, down -> residual add, next GEMM's input planes, sums of squares
//   gate/up (a CTA's tile interleaves 64 gate and 64 up features) -> silu(g) * u -> down's input planes
//   LM head -> softmax statistics per (128-token tile, row)
#pragma once

#include "sj_attn_t5.cuh"
#include "sj_gemm_tc.cuh"

namespace sj {

constexpr int kPairThreads = 384;      // warp 0 TMA, warp 1 MMA (rank 0), warp 2 tensor memory, warps 4..11 epilogue
constexpr int kPairWorkers = 256;
constexpr int kPairMaxStages = 10;
constexpr int kPairMaxRows = kMaxRows;
constexpr int kPairSegKB = 16, kPairShortKB = 32;   // K blocks of 64 per accumulation chain; half of them in a prefill's sums of up to kPairShortKB
constexpr int kPairMaxSplit = 4;        // pairs that share an item's K (a cluster of 8)
constexpr double kPairHbmBytesPerClk = 3600;   // HBM against the SM clock, for the host's choice of a geometry
constexpr int kPairXchClk = 3000;       // an exchange between the splits
__host__ __device__ constexpr int pair_chunk(bool narrow) { return narrow ? 8 : 16; }   // rows of an epilogue chunk
// "My sums have been read" barriers per epilogue group, taken in turn by successive exchanges.  A split that receives
// nothing in an exchange (all of the row block's chunks belong to others) does not wait for its partners there and may
// finish it before a partner has looked at the phase of the exchange before; on one barrier that phase would be overtaken,
// and a wait that knows only its parity would see it as not yet complete.  To finish the second exchange after, a split
// needs its partners' arrivals of the first, which they give after their look: two barriers are never overtaken.
constexpr int kPairFreeBars = 2;
constexpr uint32_t kPairSpin = kSpinLimit;

enum PairSite { PAIR_QKV = 0, PAIR_RES = 1, PAIR_GU = 2, PAIR_LM = 3 };

struct PairParams {
  int n_tiles;            // 128-feature tiles (gate/up: 64 + 64); an odd last one is paired with zeros
  int KB;                 // K blocks of 64
  int n_groups;           // clusters
  int n_split;            // pairs of a cluster: they share an item's K blocks
  int seg_kb;             // K blocks per accumulation chain
  int xch_js;             // epilogue chunks of a group that one split finishes, at most
  int R, rb, n_rb;        // rows, rows per block (a multiple of 16, at most 128: an M = 256 MMA takes N = 32, 64 .. 256), row blocks
  int plane_rows;         // row of the lo plane in the activation matrix
  int stages, stage_bytes;
  uint32_t tmem_cols;     // two accumulators of 2 rb columns
  int tile_q, tile_k;     // QKV: tiles of Wq, tiles of Wq and Wk together
  const float* ssq_in;    // [d / 128][R] sums of squares of this GEMM's input rows (null: LM head, whose planes are normalised)
  float* ssq_out;         // [d / 128][R] PAIR_RES
  const bf16* gain;       // PAIR_RES: gain of the norm that reads the result next
  void* planes_out;       // PAIR_RES: W.A; PAIR_GU: W.H
  int K_out;              // row length of planes_out
  int layer;
  const bf16 *bq, *bk, *bv;
};

struct PairCtl {
  uint64_t full[kPairMaxStages], empty[kPairMaxStages], tmem_full[2], tmem_empty[2];
  uint64_t xch_full[2];                  // per epilogue group: the other splits' sums are here
  uint64_t xch_free[2][kPairFreeBars];   // the others have read mine
  uint32_t tmem_base;
  int abort_flag;
  float inv[kPairMaxRows];
};
struct PairQkvCtl {
  int qoff[kPairMaxRows], nkvoff[kPairMaxRows];
  long long kvoff[kPairMaxRows];   // -1: the row is not stored
  float exch[2][128][9];
};
struct PairGuCtl { float exch[2][128][9]; };
struct PairResCtl { float sums[4][128]; };   // by row of the item's block
struct PairLmCtl {
  int tok[kPairMaxRows];
  float pre[kPairMaxRows];
  RowStat st[2][4][16];
};
template <int SITE> struct PairExtra;
template <> struct PairExtra<PAIR_QKV> { typedef PairQkvCtl type; };
template <> struct PairExtra<PAIR_RES> { typedef PairResCtl type; };
template <> struct PairExtra<PAIR_GU> { typedef PairGuCtl type; };
template <> struct PairExtra<PAIR_LM> { typedef PairLmCtl type; };
template <int SITE> struct PairSmem { PairCtl c; typename PairExtra<SITE>::type x; };

// ---- cta_group::2 wrappers -----------------------------------------------------------------------
constexpr uint32_t kPeerMask = 0xFEFFFFFFu;   // a shared::cluster address with the CTA bit cleared: the pair's rank 0
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive_all() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait_all() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all() {
  cluster_arrive_all();
  cluster_wait_all();
}
__device__ __forceinline__ void pair_tma_2d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4}], [%2], %5;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(bar & kPeerMask), "r"(c0), "r"(c1), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void pair_commit(uint32_t bar, uint32_t mask) {   // arrives on `bar` of both CTAs of the pair (mask)
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"((uint16_t)mask)
      : "memory");
}
__device__ __forceinline__ void pair_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, int cta) {   // the same shared-memory address in CTA `cta` of the cluster
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(cta));
  return remote;
}
__device__ __forceinline__ void cluster_arrive(uint32_t bar, int cta) {   // releases this warp's earlier writes to that CTA
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr(bar, cta)) : "memory");
}
__device__ __forceinline__ bool cluster_try_wait(uint32_t bar, uint32_t parity) {   // acquires what other CTAs of the cluster released
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Four values to another CTA of the cluster; their arrival counts 16 bytes on that CTA's barrier (an address there).
__device__ __forceinline__ void cluster_st4_async(uint32_t remote, const float* v, uint32_t remote_bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(remote), "f"(v[0]), "f"(v[1]),
               "f"(v[2]), "f"(v[3]), "r"(remote_bar)
               : "memory");
}
__device__ __forceinline__ uint32_t instr_desc_pair(int n) {   // M = 256
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
}

// NARROW: row blocks of 16, whose rows the two epilogue groups halve (chunks of 8 rows).  With chunks of 16 the second group had
// nothing to do and every slot of 16 issued for the 5 rows of a toy step (68.1 -> 52.8 us, two caches in turn; alone 128 -> 114, B200).  Wider blocks keep chunks of 16: with 8
// a score of 44 rows was 3 % slower.
template <int SITE, int HD, bool NARROW>
static __global__ void __launch_bounds__(kPairThreads, 1)
k_gemm_pair(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW0, const __grid_constant__ CUtensorMap tmW1,
            const __grid_constant__ CUtensorMap tmW2, const PairParams p, const StepArgs* __restrict__ args, const KvView kv, const Work w,
            const Dims dm) {
  // rows of an epilogue chunk, chunks of a group, lanes that share a row's totals
  constexpr int CH = pair_chunk(NARROW), NJ = NARROW ? 1 : 4, LPR = 32 / CH;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  // ring | the other splits' sums [n_split - 1][2 groups][xch_js][CH / 4][128 features] of 4 rows each | control
  float4* xch = reinterpret_cast<float4*>(smem + (size_t)p.stages * p.stage_bytes);
  PairSmem<SITE>* sm = reinterpret_cast<PairSmem<SITE>*>(xch + (size_t)(p.n_split - 1) * 2 * p.xch_js * (32 * CH));
  PairCtl* ctl = &sm->c;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int S = p.n_split, crank = (int)cluster_rank(), rank = crank & 1, split = crank >> 1, g = blockIdx.x / (2 * S);
  const int kb_lo = p.KB * split / S, kb_hi = p.KB * (split + 1) / S;   // this pair's K blocks
  const uint32_t pair_mask = 3u << (crank & ~1);
  volatile int* abort_flag = &ctl->abort_flag;
  const int n_items = (p.n_tiles + 1) / 2 * p.n_rb;

  if (threadIdx.x == 0) {
    for (int i = 0; i < p.stages; ++i) {
      mbar_init(smem_u32(&ctl->full[i]), 1);
      mbar_init(smem_u32(&ctl->empty[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&ctl->tmem_full[i]), 1);
      mbar_init(smem_u32(&ctl->tmem_empty[i]), 16);   // the epilogue warps of both CTAs
      mbar_init(smem_u32(&ctl->xch_full[i]), 1);   // and the bytes of the other splits' sums
      for (int k = 0; k < kPairFreeBars; ++k) mbar_init(smem_u32(&ctl->xch_free[i][k]), 4 * max(S - 1, 1));   // a group's warps of every other split
    }
    ctl->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)), "r"(p.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // the other CTA's barriers exist
  tc_fence_after();
  pdl_launch();
  const uint32_t tmem_base = ctl->tmem_base;

  if (warp == 0) {
    // ------------------------------ TMA producer (both CTAs) ------------------------------
    if (elect_one()) {
      const uint64_t pol_w = l2_policy_evict_first(), pol_a = l2_policy_evict_last();
      const uint32_t tx = 2u * (kWTileBytes + (uint32_t)p.rb * 128u);   // both CTAs' bytes land on rank 0's barrier
      auto w_load = [&](int s, int tile2, int kb) {
        const int tile = 2 * tile2 + rank;
        const uint32_t bar = smem_u32(&ctl->full[s]), dst = smem_u32(smem + (size_t)s * p.stage_bytes);
        if (rank == 0) mbar_expect_tx(bar, tx);
        if (SITE == PAIR_GU) {
          pair_tma_2d(dst, &tmW0, bar, kb * kBK, tile * 64, pol_w);
          pair_tma_2d(dst + 8192u, &tmW1, bar, kb * kBK, tile * 64, pol_w);
        } else if (SITE == PAIR_QKV) {
          if (tile < p.tile_q) pair_tma_2d(dst, &tmW0, bar, kb * kBK, tile * kTileN, pol_w);
          else if (tile < p.tile_k) pair_tma_2d(dst, &tmW1, bar, kb * kBK, (tile - p.tile_q) * kTileN, pol_w);
          else pair_tma_2d(dst, &tmW2, bar, kb * kBK, (tile - p.tile_k) * kTileN, pol_w);
        } else {
          pair_tma_2d(dst, &tmW0, bar, kb * kBK, tile * kTileN, pol_w);
        }
      };
      // the first ring-full of weights before the programmatic wait: they do not depend on the previous kernel
      int pre = 0;
      for (int item = g; item < n_items && pre < p.stages; item += p.n_groups)
        for (int kb = kb_lo; kb < kb_hi && pre < p.stages; ++kb) w_load(pre++, item / p.n_rb, kb);
      pdl_wait();
      int s = 0, r = 0;
      bool alive = true;
      for (int item = g; item < n_items && alive; item += p.n_groups) {
        const int tile2 = item / p.n_rb, row = rank * p.plane_rows + (item % p.n_rb) * p.rb;
        for (int kb = kb_lo; kb < kb_hi; ++kb) {
          if (r > 0) {
            if (!mbar_wait(smem_u32(&ctl->empty[s]), (uint32_t)(r - 1) & 1u, abort_flag, w.status, kPairSpin)) { alive = false; break; }
            w_load(s, tile2, kb);
          }
          pair_tma_2d(smem_u32(smem + (size_t)s * p.stage_bytes + kWTileBytes), &tmA, smem_u32(&ctl->full[s]), kb * kBK, row, pol_a);
          if (++s == p.stages) { s = 0; ++r; }
        }
      }
    } else {
      pdl_wait();
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer (rank 0) ------------------------------
    pdl_wait();
    if (rank == 0 && elect_one()) {
      const uint32_t idesc = instr_desc_pair(2 * p.rb);
      int s = 0, r = 0, n = 0;
      bool alive = true;
      for (int item = g; item < n_items && alive; item += p.n_groups) {
        uint32_t dcol = 0;
        int acc = 0, at = 0;   // block of the chain
        for (int kb = kb_lo; kb < kb_hi; ++kb) {
          const bool first = at == 0;
          if (first) {
            acc = n & 1;
            const int use = n >> 1;
            ++n;
            if (use > 0 && !mbar_wait(smem_u32(&ctl->tmem_empty[acc]), (uint32_t)(use - 1) & 1u, abort_flag, w.status, kPairSpin)) { alive = false; break; }
            dcol = tmem_base + (uint32_t)(acc * 2 * p.rb);
          }
          if (!mbar_wait(smem_u32(&ctl->full[s]), (uint32_t)r & 1u, abort_flag, w.status, kPairSpin)) { alive = false; break; }
          tc_fence_after();
          const uint32_t wa = smem_u32(smem + (size_t)s * p.stage_bytes);
          const uint64_t dw = smem_desc_sw128(wa), da = smem_desc_sw128(wa + kWTileBytes);
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k) pair_mma(dcol, dw + 2 * k, da + 2 * k, idesc, (!first || k > 0) ? 1u : 0u);
          pair_commit(smem_u32(&ctl->empty[s]), pair_mask);
          if (++s == p.stages) { s = 0; ++r; }
          if (++at == p.seg_kb || kb == kb_hi - 1) {
            pair_commit(smem_u32(&ctl->tmem_full[acc]), pair_mask);
            at = 0;
          }
        }
      }
    }
  } else if (warp >= 4) {
    // ------------------------------ epilogue (eight warps) ------------------------------
    // two groups of four warps take alternate chunks of CH rows; a warp reads the accumulator lanes 32 * (warp % 4) .. + 31
    pdl_wait();
    const int wt = threadIdx.x - 128, grp = wt >> 7, fl = wt & 127, quarter = fl >> 5, bar_id = 2 + grp;
    const int R = p.R, rows = args->gamma + 1;
    auto group_sync = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(bar_id) : "memory"); };
    auto all_sync = [&]() { asm volatile("bar.sync 1, 256;" ::: "memory"); };
    // per-row tables, beside the first MMAs
    const int nt128 = dm.d / kTileN;
    for (int r = wt; r < R; r += kPairWorkers) {
      float inv = 1.f;
      if (p.ssq_in) {
        float s = 0.f;
#pragma unroll 8
        for (int t = 0; t < nt128; ++t) s += __ldcg(p.ssq_in + (size_t)t * R + r);
        inv = 1.0f / sqrtf(s / (float)dm.d + dm.eps);
      }
      ctl->inv[r] = inv;
      if constexpr (SITE == PAIR_QKV) {
        const int b = r / rows, j = r % rows, pos = __ldcg(w.row_pos + r);
        sm->x.qoff[r] = (b * dm.Hq * rows + j) * HD;
        sm->x.nkvoff[r] = (b * dm.Hkv * 2 * rows + j) * HD;
        long long off = -1;
        if (r < args->kv_rows) {
          const int page = kv.block_table[(size_t)args->seq_ids[b] * kv.max_pages_per_seq + pos / kv.page_size];
          off = ((long long)page * 2 * dm.Hkv * kv.page_size + pos % kv.page_size) * HD;
        }
        sm->x.kvoff[r] = off;
      }
      if constexpr (SITE == PAIR_LM) {
        const int b = r / rows, j = r % rows;
        sm->x.tok[r] = j < args->gamma ? args->draft_ids[b * args->gamma + j] : -1;
        sm->x.pre[r] = args->top_k >= 2 ? __ldcg(w.tgt_pre + r) : 0.f;
      }
    }
    all_sync();
    const int n_seg = (kb_hi - kb_lo + p.seg_kb - 1) / p.seg_kb;
    float invT = 1.f, *dbg = nullptr, *keep = nullptr;
    bool topk = false;
    if constexpr (SITE == PAIR_LM) {
      invT = args->inv_temperature;
      topk = args->top_k >= 2;
      dbg = args->dbg_logits;
      keep = w.logits;
    }
    int n = 0, n_x = 0;   // segments, exchanges so far
    uint32_t mine = 0;    // the chunks j that this split finishes
    for (int j = split; j < NJ; j += S) mine |= 1u << j;
    for (int item = g; item < n_items; item += p.n_groups) {
      const int tile = 2 * (item / p.n_rb) + rank, r_lo = item % p.n_rb * p.rb, r_hi = min(r_lo + p.rb, R);
      const bool real = tile < p.n_tiles;   // an odd last tile's partner has no features
      // per-feature constants, requested beside the MMAs
      int kind = 0, head = 0, dim = 0;
      float bias = 0.f, gn = 1.f;
      if constexpr (SITE == PAIR_QKV) {
        int fs = tile * kTileN + fl;
        const bf16* bp = p.bq;
        if (tile >= p.tile_k) { kind = 2; fs -= p.tile_k * kTileN; bp = p.bv; }
        else if (tile >= p.tile_q) { kind = 1; fs -= p.tile_q * kTileN; bp = p.bk; }
        head = fs / HD;
        dim = fs % HD;
        if (bp && real) bias = __bfloat162float(bp[fs]);
      }
      if constexpr (SITE == PAIR_RES) gn = real ? __bfloat162float(p.gain[tile * kTileN + fl]) : 0.f;
      // residual rows of the first chunk that this split finishes, requested beside the MMAs
      float x_first[CH];
      if constexpr (SITE == PAIR_RES) {
#pragma unroll
        for (int i = 0; i < CH; ++i)
          x_first[i] = __ldcg(w.X + (size_t)min(r_lo + CH * (grp + 2 * split) + i, R - 1) * dm.d + min(tile, p.n_tiles - 1) * kTileN + fl);
      }
      // the segments' sums: chunk j of this group in registers
      float sum[NJ][CH];
#pragma unroll
      for (int j = 0; j < NJ; ++j)
#pragma unroll
        for (int i = 0; i < CH; ++i) sum[j][i] = 0.f;
#pragma unroll 1
      for (int sg = 0; sg < n_seg; ++sg, ++n) {
        const int acc = n & 1;
        // a wait that runs out raises the abort flag and the epilogue goes on with whatever it reads: every thread
        // keeps taking the same barriers, and the status word tells the host
        if (fl == 0) mbar_wait(smem_u32(&ctl->tmem_full[acc]), (uint32_t)(n >> 1) & 1u, abort_flag, w.status, kPairSpin);
        group_sync();
        tc_fence_after();
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * 2 * p.rb);
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          const int c = CH * (grp + 2 * j);   // row of the chunk within the block
          if (r_lo + c < r_hi) {              // uniform over the group
            float hi[CH], lo[CH];
            if constexpr (NARROW) {
              tc_ld8(taddr + (uint32_t)c, hi);
              tc_ld8(taddr + (uint32_t)(p.rb + c), lo);
            } else {
              tc_ld16(taddr + (uint32_t)c, hi);
              tc_ld16(taddr + (uint32_t)(p.rb + c), lo);
            }
#pragma unroll
            for (int i = 0; i < CH; ++i) sum[j][i] += hi[i] + lo[i];
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) cluster_arrive(smem_u32(&ctl->tmem_empty[acc]), crank & ~1);
      }
      if (S > 1) {   // send the sums that others finish, add theirs to mine
        auto xch_wait = [&](uint64_t* bar, uint32_t parity) {
          if (fl == 0) mbar_wait(smem_u32(bar), parity, abort_flag, w.status, kPairSpin);
          group_sync();
          cluster_try_wait(smem_u32(bar), parity);   // every thread acquires the completed phase
        };
        if (fl == 0) {
          uint32_t bytes = 0;
          for (int j = split; j < NJ; j += S)
            if (r_lo + CH * (grp + 2 * j) < r_hi) bytes += (uint32_t)(S - 1) * (512u * CH);
          mbar_expect_tx(smem_u32(&ctl->xch_full[grp]), bytes);
        }
        if (n_x > 0) xch_wait(&ctl->xch_free[grp][(n_x - 1) % kPairFreeBars], (uint32_t)((n_x - 1) / kPairFreeBars) & 1u);
#pragma unroll
        for (int j = 0; j < NJ; ++j)
          if (!(mine >> j & 1u) && r_lo + CH * (grp + 2 * j) < r_hi) {
            const int f = j % S, slot = split < f ? split : split - 1;
            const uint32_t dst = cluster_addr(smem_u32(xch + ((size_t)(slot * 2 + grp) * p.xch_js + j / S) * (32 * CH) + fl), 2 * f + rank);
            const uint32_t bar = cluster_addr(smem_u32(&ctl->xch_full[grp]), 2 * f + rank);
#pragma unroll
            for (int q = 0; q < CH / 4; ++q) cluster_st4_async(dst + (uint32_t)q * 2048u, &sum[j][4 * q], bar);
          }
        xch_wait(&ctl->xch_full[grp], (uint32_t)n_x & 1u);
#pragma unroll
        for (int j = 0; j < NJ; ++j)
          if ((mine >> j & 1u) && r_lo + CH * (grp + 2 * j) < r_hi) {
            for (int slot = 0; slot < S - 1; ++slot) {
              const float4* src = xch + ((size_t)(slot * 2 + grp) * p.xch_js + j / S) * (32 * CH) + fl;
#pragma unroll
              for (int q = 0; q < CH / 4; ++q) {
                const float4 x = src[q * 128];
                sum[j][4 * q] += x.x; sum[j][4 * q + 1] += x.y; sum[j][4 * q + 2] += x.z; sum[j][4 * q + 3] += x.w;
              }
            }
          }
        __syncwarp();
        if (lane == 0)
          for (int f = 0; f < S; ++f)
            if (f != split) cluster_arrive(smem_u32(&ctl->xch_free[grp][n_x % kPairFreeBars]), 2 * f + rank);
        ++n_x;
      }
      // The kernel's last cluster barrier, reported to as soon as this warp is done with the other CTAs' memory and with its
      // accumulators: nobody waits for it behind the epilogue (at the kernel's end it was 0.7 us of each: 8B-shaped 44 rows, 32 layers
      // 4.37 -> 4.26 ms a step, 1B-shaped 48 rows 1024 -> 964 us, B200).  A wait that runs out holds its warp's report back itself.
      if (item + p.n_groups >= n_items) {
        tc_fence_before();
        __syncwarp();
        cluster_arrive_all();
      }

      // Not unrolled: a chunk's own copy of this code would come from L2 when the chunk is reached, and most copies run once a
      // launch.  The sums move down a chunk each time instead.  (8B-shaped, 44 rows: a score 12602 -> 12395 us; 1B-shaped, 48 rows: a
      // step 961 -> 946; 8B-shaped prefill of 1000 tokens 32.1 -> 31.5 ms; B200.)
#pragma unroll 1
      for (int j = 0; j < NJ; ++j) {
        const int c0 = r_lo + CH * (grp + 2 * j), nr = min(CH, r_hi - c0);
        if (nr <= 0 || !real) break;   // uniform over the group
        float v[CH];
#pragma unroll
        for (int i = 0; i < CH; ++i) {
          v[i] = sum[0][i];
#pragma unroll
          for (int k = 0; k + 1 < NJ; ++k) sum[k][i] = sum[k + 1][i];
        }
        if (!(mine >> j & 1u)) continue;
        float xs[CH];
        if constexpr (SITE == PAIR_RES) {
          if (j == split) {
#pragma unroll
            for (int i = 0; i < CH; ++i) xs[i] = x_first[i];
          } else
#pragma unroll
          for (int i = 0; i < CH; ++i) xs[i] = __ldcg(w.X + (size_t)min(c0 + i, R - 1) * dm.d + tile * kTileN + fl);
        }
        if constexpr (SITE == PAIR_QKV) {
          constexpr int half = HD / 2;
#pragma unroll
          for (int i = 0; i < CH; ++i) v[i] = v[i] * (i < nr ? ctl->inv[c0 + i] : 0.f) + bias;
          if (kind < 2) {   // uniform over the CTA
#pragma unroll
            for (int h8 = 0; h8 < CH; h8 += 8) {
              float2 cs[8];
#pragma unroll
              for (int i = 0; i < 8; ++i) cs[i] = __ldcg(w.rope + (size_t)min(c0 + h8 + i, R - 1) * half + (dim & (half - 1)));
#pragma unroll
              for (int i = 0; i < 8; ++i) sm->x.exch[grp][fl][i] = v[h8 + i];
              group_sync();
              const bool lower = dim < half;
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const float xp = sm->x.exch[grp][fl ^ half][i];
                v[h8 + i] = lower ? v[h8 + i] * cs[i].x - xp * cs[i].y : v[h8 + i] * cs[i].x + xp * cs[i].y;
              }
              group_sync();
            }
          }
          if (kind == 0) {
            const float qscale = 1.4426950408889634f / sqrtf((float)HD);
            __half* qb = w.Qb + (size_t)head * rows * HD + dim;
            __half* ql = w.Qlo + (size_t)head * rows * HD + dim;
#pragma unroll
            for (int i = 0; i < CH; ++i)
              if (i < nr) {
                const float qv = v[i] * qscale;
                const __half hq = __float2half_rn(qv);
                qb[sm->x.qoff[c0 + i]] = hq;
                ql[sm->x.qoff[c0 + i]] = __float2half_rn(qv - __half2float(hq));
              }
          } else {
            bf16* kvb = reinterpret_cast<bf16*>(kv.pool) +
                        ((size_t)p.layer * kv.n_pages * 2 * dm.Hkv + (size_t)(kind - 1) * dm.Hkv + head) * kv.page_size * HD + dim;
            __half* kn = w.KVn + (size_t)(head * 2 + kind - 1) * rows * HD + dim;
#pragma unroll
            for (int i = 0; i < CH; ++i)
              if (i < nr) {
                if (sm->x.kvoff[c0 + i] >= 0) kvb[sm->x.kvoff[c0 + i]] = __float2bfloat16_rn(v[i]);
                kn[sm->x.nkvoff[c0 + i]] = __float2half_rn(v[i]);
              }
          }
        } else if constexpr (SITE == PAIR_RES) {
          const int f = tile * kTileN + fl;
          float sq[CH];
#pragma unroll
          for (int i = 0; i < CH; ++i) {
            sq[i] = 0.f;
            if (i < nr) {
              const float x = xs[i] + v[i];
              w.X[(size_t)(c0 + i) * dm.d + f] = x;
              store_act<bf16>(p.planes_out, R, dm.d, c0 + i, f, x * gn);
              sq[i] = x * x;
            }
          }
          const float t = warp_sum_n<CH>(sq, lane);
          if (lane % LPR == 0) sm->x.sums[quarter][c0 - r_lo + lane / LPR] = t;
        } else if constexpr (SITE == PAIR_GU) {
#pragma unroll
          for (int i = 0; i < CH; ++i) v[i] *= (i < nr ? ctl->inv[c0 + i] : 0.f);
          // gate threads finish the chunk's first half, up threads the second: each hands over its other values
          constexpr int H = CH / 2;
          const bool is_gate = fl < 64;
#pragma unroll
          for (int i = 0; i < H; ++i) sm->x.exch[grp][fl][i] = is_gate ? v[H + i] : v[i];
          group_sync();
          const int f = tile * 64 + (fl & 63), h8 = is_gate ? 0 : H;
#pragma unroll
          for (int i = 0; i < H; ++i) {
            const float other = sm->x.exch[grp][fl ^ 64][i];
            const float gt = is_gate ? v[i] : other, up = is_gate ? other : v[H + i];
            if (h8 + i < nr) store_act<bf16>(p.planes_out, R, p.K_out, c0 + h8 + i, f, gt / (1.0f + expf(-gt)) * up);
          }
          group_sync();
        } else {   // LM head
          // What bounds a wide step's LM head is this code's instruction count: two warps on a scheduler issue one instruction in five
          // clocks each, and at 342 rows an item's epilogue took longer than its MMAs (8B-shaped, 8 layers, top-2 alignment: a step 3607 -> 3559 us, B200).  So what concerns few steps or few
          // tiles (bounds, stored logits, drafted tokens) is decided once a chunk, and a maximum's token comes from a ballot.
          const int n_id = tile * kTileN + fl, n_warp = n_id - lane;
          const int own = lane / LPR;   // the chunk's row whose totals this lane ends up with
          if (nr < CH || (tile + 1) * kTileN > dm.V) {   // uniform over the group
#pragma unroll
            for (int i = 0; i < CH; ++i)
              if (i >= nr || n_id >= dm.V) v[i] = -INFINITY;
          }
          if (dbg || keep) {   // logits asked for; sampling mode
#pragma unroll
            for (int i = 0; i < CH; ++i)
              if (i < nr && n_id < dm.V) {
                if (dbg) dbg[(size_t)(c0 + i) * dm.V + n_id] = v[i];
                if (keep) keep[(size_t)(c0 + i) * dm.V + n_id] = v[i];
              }
          }
          // lane i (and i + CH ..): the drafted token of row i
          const int tok = lane % CH < nr ? sm->x.tok[c0 + lane % CH] : -1;
          int before = 0;
          if (topk) {   // uniform
#pragma unroll
            for (int i = 0; i < CH; ++i) {
              const int tg = __shfl_sync(0xffffffffu, tok, i);
              const float zd = sm->x.pre[min(c0 + i, R - 1)];
              const int c = __popc(__ballot_sync(0xffffffffu, n_id != tg && (v[i] > zd || (v[i] == zd && n_id < tg))));
              if (i == own && tg >= 0) before = c;
            }
          }
          if (invT != 1.f) {
#pragma unroll
            for (int i = 0; i < CH; ++i) v[i] *= invT;
          }
          const unsigned here = __ballot_sync(0xffffffffu, lane < CH && tok >= n_warp && tok < min(n_warp + 32, dm.V));
          if (here) {   // uniform over the warp: some row's drafted token is one of its tokens
#pragma unroll
            for (int i = 0; i < CH; ++i)
              if ((here >> i & 1u) && n_id == __shfl_sync(0xffffffffu, tok, i)) w.tgt_logit[c0 + i] = v[i];
          }
          const float m = warp_fmax_n<CH>(v, lane);
          int arg = 0x7fffffff;
#pragma unroll
          for (int i = 0; i < CH; ++i) {
            const float mi = __shfl_sync(0xffffffffu, m, LPR * i);
            const unsigned at = __ballot_sync(0xffffffffu, v[i] == mi);   // the lowest lane has the lowest token
            if (i == own && at) arg = n_warp + __ffs(at) - 1;
            v[i] = v[i] == -INFINITY ? 0.f : expf(v[i] - mi);
          }
          const float e = warp_sum_n<CH>(v, lane);
          if (lane % LPR == 0) {
            RowStat st; st.m = m; st.s = e; st.arg = arg; st.pad = before;
            sm->x.st[grp][quarter][own] = st;
          }
          group_sync();
          if (fl < nr) {
            RowStat a = sm->x.st[grp][0][fl];
            a = stat_merge(a, sm->x.st[grp][1][fl]);
            a = stat_merge(a, sm->x.st[grp][2][fl]);
            a = stat_merge(a, sm->x.st[grp][3][fl]);
            w.stats[(size_t)tile * R + c0 + fl] = a;
          }
          group_sync();
        }
      }
      if constexpr (SITE == PAIR_RES) {
        all_sync();
        if (real)
          for (int r = r_lo + wt; r < r_hi; r += kPairWorkers)
            if (mine >> ((r - r_lo) / (2 * CH)) & 1u)
              p.ssq_out[(size_t)tile * R + r] = (sm->x.sums[0][r - r_lo] + sm->x.sums[1][r - r_lo]) + (sm->x.sums[2][r - r_lo] + sm->x.sums[3][r - r_lo]);
        all_sync();
      }
    }
  } else {
    pdl_wait();
  }
  __syncwarp();
  if (warp < 4) {
    tc_fence_before();
    cluster_arrive_all();
  }
  cluster_wait_all();   // nothing of the pair touches the other CTA's memory after this
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(p.tmem_cols) : "memory");
  }
}

}  // namespace sj
