// Attention of the verification step on the 5th-generation tensor cores (head dimension 128, bf16 cache), split along
// the keys over all SMs like sj_attn_tc.cuh's, with both contractions on tcgen05.mma, transposed: the KEYS are the rows.
//
// One work tile is 128 cached keys of one (sequence, KV head): K and V of its 8 pages arrive by TMA (boxes of 16 slots x
// 64 dims, 128-byte swizzle) as two 32 KiB shared-memory tiles laid out [half of the head dim][page][16 keys x 128 B].
//   S^T = K Q^T   M = 128 keys, N = 2 NQ, K = head dim.  The query rows of the KV head's group (padded to NQ, a multiple
//                 of 8) are the N operand twice: as bf16 the cache's queries need two terms (16 significant bits), hi in
//                 columns [0, NQ), lo in [NQ, 2 NQ); the two scores are added when they are read.
//   softmax       thread = key (TMEM lane): it reads its key's scores of all queries, so every thread has work however few
//                 queries there are, and a tile needs no cross-lane traffic: the per-query stabiliser m is shared by the
//                 block and only moves when some score exceeds it by more than 2^16 (a vote per tile; the probabilities
//                 keep their relative precision whatever their size), and the sums of a query are per thread until the
//                 segment ends.  P goes to shared memory as bf16 hi | lo columns [128 keys][2 NQ].
//   O^T += V^T P  M = 128 dims, N = 2 NQ, K = 128 keys; V straight from the page layout (MN-major A operand), P MN-major
//                 as well.  O^T has the dims in the lanes: the segment's partial is stored coalesced.
// 16 MMAs of N = 2 NQ per tile.  With the query rows as M = 128 (the kernel before this one) 36 rows of a group of four
// heads and gamma 8 left 72 % of the accumulator lanes and softmax lanes idle and the softmax took 2060 clocks a tile,
// where HBM delivers one in 2600 to every SM; a layer of 32 sequences of 512 to 8192 keys and 8 KV
// heads (570 MB, 86 us at the copy rate) took 153 us, with this one 127 us (B200).
//
// A segment (the block's run of tiles of one (sequence, KV head)) ends with the unnormalised partial (m, l, o) per query
// row, in the format of sj_attn_tc.cuh, whose combine pass merges them; the block's own gamma+1 rows (the causal tail)
// are handled with that file's mma.sync routine, by a warp of their own beside the tiles.
//
// Every wait is bounded; one that runs out raises the abort flag, after which all others return at once: the flow goes
// on to its end with whatever it reads (named barriers are met by every warp), and the status word tells the host.
#pragma once

#include "sj_attn_tc.cuh"
#include "sj_gemm_tc.cuh"

namespace sj {

constexpr int kT5Keys = 128;               // keys per tile
constexpr int kT5Pad = 2;                  // empty tiles the plan counts per (sequence, KV head): what a segment costs a block beyond its tiles
constexpr int kT5Threads = 384;            // warp 0 key tiles, warp 10 value tiles, warp 1 MMA, warps 2..9 softmax, warp 11 the causal tails
constexpr int kT5MaxRows = 128;
constexpr uint32_t kT5Part = 32768;        // bytes of a key tile or a value tile: a ring stage
constexpr int kA5TmemCols = 512;
constexpr float kA5Raise = 16.f;           // log2: how far a score may exceed the stabiliser

__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tc_ld8_nowait(uint32_t taddr, float* v) {   // results valid after tc_wait_ld()
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tc_st8f(uint32_t taddr, const float* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(__float_as_uint(v[0])),
               "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])),
               "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7]))
               : "memory");
}

// Shared-memory descriptor of an MN-major operand in the [half][page][16 x 128 B] layout: 16 keys (one page) by
// 128 dims; the two 64-dim halves are `half_stride` bytes apart, the two 8-key groups 1024 bytes.
__device__ __forceinline__ uint64_t smem_desc_mn_sw128(uint32_t saddr, uint32_t half_stride) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)((half_stride >> 4) & 0x3FFF) << 16;   // leading byte offset: along the contiguous (head) dimension
  d |= (uint64_t)(1024 >> 4) << 32;                     // stride byte offset: along the keys
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
// bf16 x bf16 -> fp32, M = 128, N = n; a_mn / b_mn: the operand is MN-major
__device__ __forceinline__ uint32_t instr_desc_bf16_mn(int n, int a_mn, int b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Whether any of the 128 threads of named barrier `id` says so; synchronises them.
__device__ __forceinline__ bool bar_any128(int id, bool x) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.or.pred q, %2, 128, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)x), "r"(id)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ void bar_sync128(int id) { asm volatile("barrier.cta.sync %0, 128;" ::"r"(id) : "memory"); }

// ---- geometry ------------------------------------------------------------------------------------
__host__ __device__ __forceinline__ int a5_nq(int nq) { return (nq + 7) & ~7; }                                  // NQ
__host__ __device__ __forceinline__ int a5_s_bufs(int nq) { return 6 * a5_nq(nq) <= kA5TmemCols ? 2 : 1; }      // score buffers beside O^T
__host__ __device__ __forceinline__ int a5_q_area_bytes(int nq) { return 2 * 2 * a5_nq(nq) * 128; }             // two 64-dim halves of 2 NQ rows
__host__ __device__ __forceinline__ int a5_p_bytes(int nq) { return (2 * a5_nq(nq) + 63) / 64 * 16384; }        // atoms of 64 columns x 128 keys
// The two groups of 128 softmax threads split the queries: group 0 takes [0, a5_split), group 1 the rest.
__host__ __device__ __forceinline__ int a5_split(int nq) { return (a5_nq(nq) / 8 + 1) / 2 * 8; }

struct A5Bars {
  uint64_t s_full[2];   // one arrival: the issuer's commit after the score MMAs
  uint64_t s_free[2];   // 256 arrivals: the softmax threads have read the scores
  uint64_t p_full;      // 256 arrivals: the probabilities are in shared memory
  uint64_t o_done;      // one arrival: the issuer's commit after the output MMAs
  uint64_t q_ready;     // 256 arrivals
};
struct alignas(16) A5Smem {   // softmax state in shared memory, read four floats at a time
  float m[kT5MaxRows];          // stabiliser per query
  float f[kT5MaxRows];          // the factor of its last move
  float red[4][kT5MaxRows];     // per lane quarter
  int claimed;                  // value stages the first producer warp has claimed
};
__device__ __forceinline__ void a5_bars_init(A5Bars* b) {
  for (int i = 0; i < 2; ++i) {
    att_mbar_init(att_smem_u32(&b->s_full[i]), 1);
    att_mbar_init(att_smem_u32(&b->s_free[i]), 256);
  }
  att_mbar_init(att_smem_u32(&b->p_full), 256);
  att_mbar_init(att_smem_u32(&b->o_done), 1);
  att_mbar_init(att_smem_u32(&b->q_ready), 256);
}
static_assert(alignof(A5Smem) == 16 && sizeof(float) * kT5MaxRows % 16 == 0, "float4 reads of the softmax state");
struct A5Ring {
  uint64_t* full;    // [stages], one arrival
  uint64_t* empty;   // [stages], one arrival
  uint8_t* base;
  int stages;
  volatile int* abort_flag;
  int* status;
};
struct A5Pos {
  int s, r;
  __device__ __forceinline__ void next(int NS) {
    if (++s == NS) { s = 0; ++r; }
  }
};
// A tile's ring entries: the key tile (0) and the value tile (1).
struct A5Entry {
  int s[2];
  uint32_t par[2], a[2];   // stage, parity of this use, address
};
__device__ __forceinline__ A5Entry a5_entry(const A5Ring& rg, A5Pos& pos) {   // the tile at pos; pos moves past it
  A5Entry e;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    e.s[i] = pos.s;
    e.par[i] = (uint32_t)pos.r & 1u;
    e.a[i] = att_smem_u32(rg.base + (size_t)pos.s * kT5Part);
    pos.next(rg.stages);
  }
  return e;
}
__device__ __forceinline__ bool a5_wait(const A5Ring& rg, uint64_t* bar, uint32_t parity, int where, int extra) {
  return att_mbar_wait(att_smem_u32(bar), parity, rg.abort_flag, rg.status, nullptr, where, extra);
}
// The block's run of real tiles at tile t: (sequence, KV head, first tile), its length n, and nv, the same with the
// plan's empty tiles; n == 0 when only empty tiles of that (sequence, KV head) fell to this block.
__device__ __forceinline__ void a5_run_at(const AttPlan& pl, int B, long long t, long long t_hi, AttTile& x, int& n, int& nv) {
  x = att_locate(pl, B, kT5Keys, (int)t);
  nv = (int)min((long long)(x.nt_b - x.ti), t_hi - t);
  n = max(0, min(nv, x.nt_real - x.ti));
}

// The TMA loads of the block's tiles [t_lo, t_hi) of one layer, by two warps (all 32 lanes of each in the same control
// flow).  A key or value tile is sixteen boxes of 2 KiB (16 keys x 64 dims: a page's slots, one swizzle span wide), one
// per lane (half = lane / 8, page = lane % 8); sixteen lanes get theirs out in 1250 clocks, so one warp for both would
// take longer than HBM needs for the bytes.  The first warp claims every stage in ring order and loads the key tiles; it
// hands a value stage over by a count in shared memory (`claimed`: value stages claimed so far).  The
// second warp may not wait on the stages' barriers itself: key stages are freed ahead of value stages, and a warp that is
// lapped waits for a parity that has passed.  pages: the block's page ids, eight per tile (clamped to the sequence's last
// page), for its first kAttPageCache / 8 tiles.
__device__ __forceinline__ bool a5_produce(const A5Ring& rg, A5Pos& pos, const CUtensorMap* tmKV, const KvView& kv,
                                           const StepArgs* __restrict__ args, const AttPlan& pl, int B, int layer,
                                           long long t_lo, long long t_hi, const int* pages, int lane, int which, volatile int* claimed) {
  int vals = 0;
  const int half = (lane >> 3) & 1, p = lane & 7;
#pragma unroll 1
  for (long long t = t_lo; t < t_hi; ++t) {
    const AttTile x = att_locate(pl, B, kT5Keys, (int)t);
    if (x.ti >= x.nt_real) continue;   // one of the plan's empty tiles: no ring entry
    const int seq = args->seq_ids[x.b], last_page = (x.L - 1) / 16, tb = (int)(t - t_lo);
    int pi = x.ti * 8 + p;
    if (pi > last_page) pi = last_page;   // keys there are masked; reload a valid page
    const int page = (tb + 1) * 8 <= kAttPageCache ? pages[tb * 8 + p]
                                                   : __ldg(kv.block_table + (size_t)seq * kv.max_pages_per_seq + pi);
    const long long row = ((((long long)layer * kv.n_pages + page) * 2 + which) * kv.n_kv_heads + x.h) * 16;
    ++vals;
    if (which == 1) {
      for (uint32_t i = 0; *claimed < vals; ++i) {
        if (i > 64) {
          if (*rg.abort_flag) return false;
          __nanosleep(20);
        }
        if (i >= 16 * kAttSpin) {   // polls of shared memory, far shorter than those of a barrier
          *rg.abort_flag = 1; atomicCAS(rg.status, DEV_OK, DEV_TIMEOUT); return false; }
      }
      __syncwarp();
    }
#pragma unroll 1
    for (int e = 0; e < 2; ++e) {
      const uint32_t bar = att_smem_u32(&rg.full[pos.s]);
      if (which == 0) {
        if (pos.r > 0 && !a5_wait(rg, &rg.empty[pos.s], (uint32_t)(pos.r - 1) & 1u, 1, pos.r)) return false;
        if (lane == 0) {
          att_mbar_expect_tx(bar, kT5Part);
          if (e == 1) {
            __threadfence_block();
            *claimed = vals;
          }
        }
      }
      if (e == which && lane < 16)
        att_tma_2d(att_smem_u32(rg.base + (size_t)pos.s * kT5Part) + (uint32_t)(half * 16384 + p * 2048), tmKV, bar, half * 64, (int)row);
      pos.next(rg.stages);
    }
  }
  return true;
}

// One elected thread: the MMAs of the block's tiles.  Order: scores(0) .. scores(n_s - 1), then output(i), scores(i + n_s),
// so that a tile's scores are ready while the softmax of the one before runs, and an output never waits behind scores
// whose keys have not arrived (with output(i) after scores(i + 1) a tile took 4000 clocks).  gt, segs: tiles and segments so far (advanced).  p_area: address of the probabilities.
__device__ __forceinline__ bool a5_issue(const A5Ring& rg, A5Pos& pos, A5Bars* ab, uint32_t tmem, uint32_t q_area, uint32_t p_area, int nq,
                                         const AttPlan& pl, int B, long long t_lo, long long t_hi, int& gt, int& segs) {
  const int NQ2 = 2 * a5_nq(nq), n_s = a5_s_bufs(nq);
  const uint32_t id_s = instr_desc_bf16_mn(NQ2, 0, 0), id_o = instr_desc_bf16_mn(NQ2, 1, 1);
  const uint64_t dq = smem_desc_sw128(q_area);
  const uint64_t q_half = (uint64_t)((NQ2 * 128) >> 4), k_half = (uint64_t)(16384 >> 4);   // start-address field, 16-byte units
  const uint32_t d_o = tmem + (uint32_t)(n_s * NQ2);
  long long t = t_lo;
#pragma unroll 1
  while (t < t_hi) {
    AttTile x;
    int n, nv;
    a5_run_at(pl, B, t, t_hi, x, n, nv);
    t += nv;
    if (n == 0) continue;   // only empty tiles of this (sequence, KV head): no segment
    if (!a5_wait(rg, &ab->q_ready, (uint32_t)segs & 1u, 2, segs)) return false;
    tc_fence_after();
    A5Entry pend[2];   // entries of the tiles whose scores have been issued and outputs have not: pend[i & 1]
#pragma unroll 1
    for (int i = -n_s; i < n; ++i) {
      if (i >= 0) {   // output of tile i
        const int g = gt + i;
        const A5Entry e = n_s == 2 && (i & 1) ? pend[1] : pend[0];
        if (!a5_wait(rg, &ab->p_full, (uint32_t)g & 1u, 5, g) || !a5_wait(rg, &rg.full[e.s[1]], e.par[1], 6, g)) return false;
        tc_fence_after();
        const uint64_t dv = smem_desc_mn_sw128(e.a[1], 16384u), dp = smem_desc_mn_sw128(p_area, 16384u);
#pragma unroll
        for (int k = 0; k < 8; ++k)   // 16 keys each
          tc_mma_bf16(d_o, dv + (uint64_t)(k * (2048 >> 4)), dp + (uint64_t)(k * (2048 >> 4)), id_o, (i > 0 || k > 0) ? 1u : 0u);
        tc_commit(att_smem_u32(&ab->o_done));
        tc_commit(att_smem_u32(&rg.empty[e.s[1]]));
      }
      if (i + n_s < n) {   // scores of tile i + n_s
        const A5Entry e = a5_entry(rg, pos);
        const int g = gt + i + n_s, b = n_s == 2 ? g & 1 : 0, use = n_s == 2 ? g >> 1 : g;
        if (use > 0 && !a5_wait(rg, &ab->s_free[b], (uint32_t)(use - 1) & 1u, 3, g)) return false;
        if (!a5_wait(rg, &rg.full[e.s[0]], e.par[0], 3, g)) return false;
        tc_fence_after();
        const uint64_t dk = smem_desc_sw128(e.a[0]);
        const uint32_t d_s = tmem + (uint32_t)(b * NQ2);
#pragma unroll
        for (int k = 0; k < 8; ++k)
          tc_mma_bf16(d_s, dk + (uint64_t)(k >> 2) * k_half + (uint64_t)(2 * (k & 3)), dq + (uint64_t)(k >> 2) * q_half + (uint64_t)(2 * (k & 3)), id_s,
                      k > 0 ? 1u : 0u);
        tc_commit(att_smem_u32(&ab->s_full[b]));
        tc_commit(att_smem_u32(&rg.empty[e.s[0]]));
        if (n_s == 2 && ((i + n_s) & 1)) pend[1] = e;
        else pend[0] = e;
      }
    }
    gt += n;
    ++segs;
  }
  return true;
}

// byte offset of (row, dim) in the query area: two K-major halves of NQ2 rows x 128 B, 128-byte swizzle
__device__ __forceinline__ uint32_t a5_q_off(int row, int dim, int NQ2) {
  return (uint32_t)((dim >> 6) * NQ2 * 128 + row * 128 + ((((dim & 63) >> 3) ^ (row & 7)) << 4));
}

// The softmax side: eight warps in two groups of 128 threads, thread = key = TMEM lane; group `grp` handles the queries
// [0, a5_split) or the rest and meets at named barrier `bar_id`.  MAXC: most 8-query chunks of a group.  The partial slot of the block's segment is slot0 + b * Hkv + h (sub-partial 0).
template <int MAXC>
__device__ __forceinline__ bool a5_softmax(const A5Ring& rg, A5Bars* ab, A5Smem* sh, uint32_t tmem, uint8_t* q_area, uint8_t* p_area,
                                           const AttArgs& a, const AttPlan& pl, int B, int Hkv, int nq, long long t_lo, long long t_hi, int& gt,
                                           int slot0, int quarter, int grp, int bar_id, int lane) {
  constexpr int HD = 128;
  const int NQ = a5_nq(nq), NQ2 = 2 * NQ, n_s = a5_s_bufs(nq), split = a5_split(nq);
  const int q0 = grp ? split : 0, nch = (grp ? NQ - split : split) / 8;
  const int key = 32 * quarter + lane;
  const uint32_t lane_addr = tmem + ((uint32_t)(32 * quarter) << 16);
  const uint32_t o_addr = lane_addr + (uint32_t)(n_s * NQ2);
  // queries of a (sequence, KV head): fp16 (plus what its rounding dropped, in the two-term layers) -> two bf16 terms
  auto deliver_q = [&](const AttTile& x) {
    const __half* qh = a.Qb + ((size_t)x.b * Hkv + x.h) * nq * HD;
    const __half* ql = a.Qlo ? a.Qlo + ((size_t)x.b * Hkv + x.h) * nq * HD : nullptr;
    const int n16 = nq * (HD / 8);
#pragma unroll 1
    for (int i0 = grp * 128 + key; i0 < n16; i0 += 4 * 256) {
      uint4 raw[4], rawl[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {   // all loads first: one at a time they cost 0.4 us each
        const int i = min(i0 + u * 256, n16 - 1);
        raw[u] = __ldcg(reinterpret_cast<const uint4*>(qh) + i);
        rawl[u] = ql ? __ldcg(reinterpret_cast<const uint4*>(ql) + i) : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * 256;
        if (i < n16) {
          const __half2* h2 = reinterpret_cast<const __half2*>(&raw[u]);
          const __half2* l2 = reinterpret_cast<const __half2*>(&rawl[u]);
          uint32_t hi[4], lo[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float2 v = __half22float2(h2[e]);
            const float2 vl = __half22float2(l2[e]);
            v.x += vl.x;
            v.y += vl.y;
            const __nv_bfloat162 bh = __floats2bfloat162_rn(v.x, v.y);
            const float2 back = __bfloat1622float2(bh);
            const __nv_bfloat162 bl = __floats2bfloat162_rn(v.x - back.x, v.y - back.y);
            hi[e] = *reinterpret_cast<const uint32_t*>(&bh);
            lo[e] = *reinterpret_cast<const uint32_t*>(&bl);
          }
          const int row = i / (HD / 8), dim = (i % (HD / 8)) * 8;
          *reinterpret_cast<uint4*>(q_area + a5_q_off(row, dim, NQ2)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          *reinterpret_cast<uint4*>(q_area + a5_q_off(NQ + row, dim, NQ2)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the MMAs read these generic-proxy stores
    att_mbar_arrive(att_smem_u32(&ab->q_ready));
  };
  long long t = t_lo;
  bool first_seg = true;
#pragma unroll 1
  while (t < t_hi) {
    AttTile x;
    int n, nv;
    a5_run_at(pl, B, t, t_hi, x, n, nv);
    const size_t base = (((size_t)slot0 + (size_t)x.b * Hkv + x.h) * kAttMaxSub + 0) * (size_t)nq;
    if (n == 0) {
      // the combine pass still reads the block's slot for this (sequence, KV head): a partial of weight zero (the
      // stored outputs are finite: old values or zeros)
      if (grp == 0 && key < nq) {
        a.P.m[base + key] = -INFINITY;
        a.P.l[base + key] = 0.f;
      }
      t += nv;
      continue;
    }
    if (first_seg) deliver_q(x);   // later segments' queries were delivered while the segment before them ended
    first_seg = false;
    float l[MAXC][8];
#pragma unroll
    for (int c = 0; c < MAXC; ++c)
#pragma unroll
      for (int e = 0; e < 8; ++e) l[c][e] = 0.f;
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      const int g = gt + i, b = n_s == 2 ? g & 1 : 0, use = n_s == 2 ? g >> 1 : g;
      a5_wait(rg, &ab->s_full[b], (uint32_t)use & 1u, 7, g);
      __syncwarp();
      tc_fence_after();
      const uint32_t s_addr = lane_addr + (uint32_t)(b * NQ2 + q0);
      float s[MAXC][8];
#pragma unroll
      for (int c = 0; c < MAXC; c += 2) {   // two chunks (four loads) at a time
        float lo[2][8];
#pragma unroll
        for (int d = 0; d < 2; ++d)
          if (c + d < nch) {   // uniform over the group
            tc_ld8_nowait(s_addr + (uint32_t)(8 * (c + d)), s[min(c + d, MAXC - 1)]);
            tc_ld8_nowait(s_addr + (uint32_t)(NQ + 8 * (c + d)), lo[d]);
          }
        tc_wait_ld();
#pragma unroll
        for (int d = 0; d < 2; ++d)
          if (c + d < nch)
#pragma unroll
            for (int e = 0; e < 8; ++e) s[min(c + d, MAXC - 1)][e] += lo[d][e];
      }
      tc_fence_before();
      att_mbar_arrive(att_smem_u32(&ab->s_free[b]));
      if (key >= x.L - (x.ti + i) * kT5Keys) {   // only in a sequence's last tile
#pragma unroll
        for (int c = 0; c < MAXC; ++c)
#pragma unroll
          for (int e = 0; e < 8; ++e) s[c][e] = -INFINITY;
      }
      // does any score outgrow its stabiliser?
      bool over = i == 0;
      if (i > 0) {
        float ex = -INFINITY;
#pragma unroll
        for (int c = 0; c < MAXC; ++c)
          if (c < nch) {
            const float4 m0 = *reinterpret_cast<const float4*>(&sh->m[q0 + 8 * c]), m1 = *reinterpret_cast<const float4*>(&sh->m[q0 + 8 * c + 4]);
            ex = fmaxf(ex, fmaxf(fmaxf(s[c][0] - m0.x, s[c][1] - m0.y), fmaxf(s[c][2] - m0.z, s[c][3] - m0.w)));
            ex = fmaxf(ex, fmaxf(fmaxf(s[c][4] - m1.x, s[c][5] - m1.y), fmaxf(s[c][6] - m1.z, s[c][7] - m1.w)));
          }
        over = bar_any128(bar_id, ex > kA5Raise);
      }
      if (over) {   // uniform over the group: the segment's first tile, and rarely later
#pragma unroll
        for (int c = 0; c < MAXC; ++c)
          if (c < nch) {
            const float mx = warp_fmax_n<8>(s[c], lane);
            if ((lane & 3) == 0) sh->red[quarter][q0 + 8 * c + (lane >> 2)] = mx;
          }
        bar_sync128(bar_id);
        if (key < 8 * nch) {
          const int q = q0 + key;
          const float old = i == 0 ? -INFINITY : sh->m[q];
          const float mn = fmaxf(old, fmaxf(fmaxf(sh->red[0][q], sh->red[1][q]), fmaxf(sh->red[2][q], sh->red[3][q])));
          sh->m[q] = mn;
          sh->f[q] = i == 0 ? 1.f : ex2_approx(old - mn);
        }
        bar_sync128(bar_id);
        if (i > 0) {   // what has been accumulated: the sums, and (once its last MMAs have completed) the output
          a5_wait(rg, &ab->o_done, (uint32_t)(g - 1) & 1u, 8, g);
          __syncwarp();
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < MAXC; ++c)
            if (c < nch) {
              float hi[8], lo[8];
              tc_ld8_nowait(o_addr + (uint32_t)(q0 + 8 * c), hi);
              tc_ld8_nowait(o_addr + (uint32_t)(NQ + q0 + 8 * c), lo);
              tc_wait_ld();
#pragma unroll
              for (int e = 0; e < 8; ++e) {
                const float f = sh->f[q0 + 8 * c + e];
                l[c][e] *= f;
                hi[e] *= f;
                lo[e] *= f;
              }
              tc_st8f(o_addr + (uint32_t)(q0 + 8 * c), hi);
              tc_st8f(o_addr + (uint32_t)(NQ + q0 + 8 * c), lo);
            }
          tc_wait_st();
        }
      }
      // the tile's place for the probabilities is free once the output MMAs that read the one before have completed
      if (i > 0) a5_wait(rg, &ab->o_done, (uint32_t)(g - 1) & 1u, 9, g);   // (every phase is waited for: a parity wait may not skip one)
      __syncwarp();
      // probabilities as two bf16 terms: hi = p truncated to bf16, lo = the rest rounded to bf16 (16 significant bits)
#pragma unroll
      for (int c = 0; c < MAXC; ++c)
        if (c < nch) {
          const float4 m0 = *reinterpret_cast<const float4*>(&sh->m[q0 + 8 * c]), m1 = *reinterpret_cast<const float4*>(&sh->m[q0 + 8 * c + 4]);
          const float mm[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
          uint32_t hi[4], lo[4];
#pragma unroll
          for (int e = 0; e < 8; e += 2) {
            const float p0 = ex2_approx(s[c][e] - mm[e]), p1 = ex2_approx(s[c][e + 1] - mm[e + 1]);   // 0 for masked keys
            l[c][e] += p0;
            l[c][e + 1] += p1;
            const uint32_t b0 = __float_as_uint(p0), b1 = __float_as_uint(p1);
            hi[e >> 1] = __byte_perm(b0, b1, 0x7632);
            const __nv_bfloat162 bl = __floats2bfloat162_rn(p0 - __uint_as_float(b0 & 0xffff0000u), p1 - __uint_as_float(b1 & 0xffff0000u));
            lo[e >> 1] = *reinterpret_cast<const uint32_t*>(&bl);
          }
          const int nh = q0 + 8 * c, nl = NQ + nh;   // columns; [64-column atom][key][128 B], 128-byte swizzle
          *reinterpret_cast<uint4*>(p_area + (nh >> 6) * 16384 + key * 128 + ((((nh & 63) >> 3) ^ (key & 7)) << 4)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          *reinterpret_cast<uint4*>(p_area + (nl >> 6) * 16384 + key * 128 + ((((nl & 63) >> 3) ^ (key & 7)) << 4)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the MMAs read these generic-proxy stores
      tc_fence_before();
      att_mbar_arrive(att_smem_u32(&ab->p_full));
    }
    // The next segment's queries, before this one is wound up: every score MMA of this segment has completed (this
    // thread saw the scores of its last tile), so the query area is free once every thread is here, and the issuer starts
    // on the next segment's scores while the partial below is read out (its first output MMAs wait for probabilities that
    // this thread delivers only afterwards, so the output accumulator is not touched early).
    for (long long t2 = t + nv; t2 < t_hi;) {
      AttTile x2;
      int n2, nv2;
      a5_run_at(pl, B, t2, t_hi, x2, n2, nv2);
      if (n2 > 0) {
        deliver_q(x2);
        break;
      }
      t2 += nv2;
    }
    // the segment's partial: (m, l, o) of every query row
#pragma unroll
    for (int c = 0; c < MAXC; ++c)
      if (c < nch) {
        const float s8 = warp_sum_n<8>(l[c], lane);
        if ((lane & 3) == 0) sh->red[quarter][q0 + 8 * c + (lane >> 2)] = s8;
      }
    bar_sync128(bar_id);
    if (key < 8 * nch && q0 + key < nq) {
      const int q = q0 + key;
      a.P.m[base + q] = sh->m[q];
      a.P.l[base + q] = (sh->red[0][q] + sh->red[1][q]) + (sh->red[2][q] + sh->red[3][q]);
    }
    {
      const int g = gt + n - 1;
      a5_wait(rg, &ab->o_done, (uint32_t)g & 1u, 9, g);
      __syncwarp();
      tc_fence_after();
      float* dst = a.P.o + (base + q0) * HD + key;   // lane == dim
#pragma unroll
      for (int c = 0; c < MAXC; ++c)
        if (c < nch) {
          float hi[8], lo[8];
          tc_ld8_nowait(o_addr + (uint32_t)(q0 + 8 * c), hi);
          tc_ld8_nowait(o_addr + (uint32_t)(NQ + q0 + 8 * c), lo);
          tc_wait_ld();
#pragma unroll
          for (int e = 0; e < 8; ++e)
            if (q0 + 8 * c + e < nq) dst[(size_t)(8 * c + e) * HD] = hi[e] + lo[e];
        }
      tc_fence_before();
    }
    bar_sync128(bar_id);   // the sums have been read before the next segment's first tile reuses their place
    gt += n;
    t += nv;
  }
  return *rg.abort_flag == 0;
}

// ---------------------------------------------------------------------------------------------
// the kernel: one block per SM
// ---------------------------------------------------------------------------------------------
constexpr int kT5MaxStages = 6;
struct T5Ctl {
  uint64_t full[kT5MaxStages], empty[kT5MaxStages];
  A5Bars bars;
  A5Smem sh;
  uint32_t tmem_base;
  int abort_flag;
  AttPlan plan;
  int pages[kAttPageCache];
};
struct T5Geom { int stages; size_t smem; };
__host__ __forceinline__ T5Geom t5_geom(int nq) {
  const size_t fixed = (size_t)a5_q_area_bytes(nq) + a5_p_bytes(nq) + sizeof(T5Ctl) + 1024;
  T5Geom g;
  g.stages = (int)((227 * 1024 - fixed) / kT5Part);
  if (g.stages > kT5MaxStages) g.stages = kT5MaxStages;
  g.smem = fixed + (size_t)g.stages * kT5Part;
  return g;
}

template <int MAXC>
static __global__ void __launch_bounds__(kT5Threads, 1)
k_attn_t5(const __grid_constant__ CUtensorMap tmKV, const StepArgs* __restrict__ args, KvView kv, Work w, Dims dm, AttArgs a, int stages) {
  constexpr int HD = 128;
  extern __shared__ uint8_t t5_smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(t5_smem_raw) + 1023) & ~(uintptr_t)1023);
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int B = args->B, rows = args->gamma + 1, Hkv = dm.Hkv, group = dm.Hq / dm.Hkv, nq = group * rows;
  const int G = gridDim.x, c = blockIdx.x;
  uint8_t* p_area = sm + (size_t)stages * kT5Part;
  uint8_t* q_area = p_area + a5_p_bytes(nq);
  T5Ctl* ctl = reinterpret_cast<T5Ctl*>(q_area + a5_q_area_bytes(nq));
  if (threadIdx.x == 0) {
    for (int i = 0; i < stages; ++i) {
      att_mbar_init(att_smem_u32(&ctl->full[i]), 1);
      att_mbar_init(att_smem_u32(&ctl->empty[i]), 1);
    }
    a5_bars_init(&ctl->bars);
    ctl->sh.claimed = 0;
    ctl->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) att_plan_fill(&ctl->plan, w.row_pos, B, rows, Hkv, kT5Keys, lane, kT5Pad);
  // padding query rows stay zero for the whole kernel
#pragma unroll 1
  for (int i = threadIdx.x; i < a5_q_area_bytes(nq) / 16; i += blockDim.x) reinterpret_cast<uint4*>(q_area)[i] = make_uint4(0, 0, 0, 0);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the MMAs read them
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(att_smem_u32(&ctl->tmem_base)), "r"((uint32_t)kA5TmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_launch();   // with this block's tensor memory in hand: a dependent that got there first would wait for this kernel, and this for it
  const AttPlan& pl = ctl->plan;
  const long long t_lo = att_first_tile(c, pl.T, G), t_hi = att_first_tile(c + 1, pl.T, G);
  att_fill_pages(ctl->pages, pl, kv, args, B, kT5Keys, t_lo, t_hi, threadIdx.x, blockDim.x);
  __syncthreads();
  const uint32_t tmem = ctl->tmem_base;
  // All of the above reads what kernels before the previous one have written.  So do the loads of the cache's tiles, but
  // in a prefill, whose entries attend to rows that the previous kernel stores.
  if (!((warp == 0 || warp == 10) && args->pos_step == 0)) pdl_wait();
  const A5Ring rg{ctl->full, ctl->empty, sm, stages, &ctl->abort_flag, w.status};
  A5Pos pos{0, 0};
  int gt = 0, segs = 0;
  if (warp == 0 || warp == 10) {
    a5_produce(rg, pos, &tmKV, kv, args, pl, B, a.layer, t_lo, t_hi, ctl->pages, lane, warp == 0 ? 0 : 1, &ctl->sh.claimed);
  } else if (warp == 1) {
    if (elect_one()) a5_issue(rg, pos, &ctl->bars, tmem, att_smem_u32(q_area), att_smem_u32(p_area), nq, pl, B, t_lo, t_hi, gt, segs);
  } else if (warp < 10) {
    const int grp = (warp - 2) >> 2;
    a5_softmax<MAXC>(rg, &ctl->bars, &ctl->sh, tmem, q_area, p_area, a, pl, B, Hkv, nq, t_lo, t_hi, gt, c, warp & 3, grp, 2 + grp, lane);
  } else {
    // the causal tails (the step's own rows as keys; mma.sync): one m-tile of one (sequence, KV head) per task, dealt
    // over all blocks from the last block down, beside the tiles
    const AttGeom g = att_geom(HD, group, rows);
    AttWarp<HD, 2> st;
#pragma unroll 1
    for (int task = G - 1 - c; task < B * Hkv * g.MT; task += G) att_tail_task<HD, 2>(st, g, a, task / g.MT, (task % g.MT) * 16, lane);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    if (*(volatile int*)&ctl->abort_flag) __nanosleep(20000);   // let copies in flight land before the block retires
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)kA5TmemCols) : "memory");
  }
}

}  // namespace sj
