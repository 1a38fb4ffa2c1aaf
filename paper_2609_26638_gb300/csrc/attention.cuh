// attention.cuh -- hybrid-mask attention over the paged fp16 KV cache, on
// the tcgen05 tensor cores.
//
// A query block is a run of at most 128 / G tokens of one sequence (a decode
// window, cut into sub-blocks when K+1 tokens carry more than 128 rows, or a
// slice of a prefill chunk); its rows are (token, query head of the GQA
// group), so the query heads that share a KV head read each K/V page once.
// Every query token carries its own inclusive key limit, which encodes the
// mask: draft boundary row n, draft mask rows n+K, verify row i n+1+i, prefill
// row p (paper Appendix steps Draft forward / Verify forward).
//
// Work items.  The block's pages are cut into fixed absolute ranges of SP
// pages ("items"): item i covers pages [i*SP, (i+1)*SP); one CTA reduces one
// item, pages in order.  A page holds K as [64 tokens][64 dims] and V
// transposed, [64 dims][64 tokens] (8 KB each), so both are K-major operands.
// Per page j:
//   S_j = Q K_j^T       tcgen05.mma M=128 (rows) N=64 (keys) K=64 into TMEM
//   softmax             per row: running max m (log2 units), P_j =
//                       exp2(s*scale - m) as fp16 into shared memory (the A
//                       operand of the next MMA)
//   O += P_j [V_j | 1]  tcgen05.mma M=128 N=80 K=64 (keys), O in TMEM: 64 dims
//                       and, from 16 rows of ones kept after every V^T page,
//                       the row sum l in O's column 64 (fp32 on the tensor core)
// The max only moves when a page raises it by more than 2^8: then the thread
// first rescales its O row in TMEM (and l with it) by exp2(m_old - m_new).  Smaller
// rises keep the old m, so P stays <= 2^8 (well inside fp16).  Either way
// O / l is the softmax-weighted sum.  Block row rr sits in MMA row (TMEM lane)
// 32 (rr mod 4) + rr / 4, so warps 0-3 (one lane quarter each) hold a quarter
// of the rows each, whatever their number; warp 4 streams K/V pages by TMA
// (128-byte swizzle) through a ring of stages; warp 5 issues the MMAs, S one
// page ahead of the softmax, S double-buffered.
//
// Merge over items, item order 0, 1, ...: M = max m_i, w_i = exp2(m_i - M),
// coef_i = w_i / sum_j w_j l_j, O = sum coef_i O_i.  A block with one item
// writes its rows directly.  The kernel of this file is for small launches (at
// most 16 items per (block, head), about one wave of CTAs; two waves for at most
// eight items of more than 96 rows): the items of a
// (block, head) form a thread-block cluster, and once every CTA of it has
// finished its pages, each sends the rows that CTA (r mod n) owns to it with one
// bulk async copy into its shared memory, completing on its mbarrier, and each
// owner merges its rows.  Larger launches run attention_stream.cuh: there every
// item writes its rows to global scratch and the last one to finish (atomic
// ticket per (block, head), no spinning) merges them.  Both run the same
// arithmetic in the same order.
//
// Invariance.  Item boundaries are absolute page numbers fixed by SP, pages
// are reduced in order, the MMA's arithmetic for a row does not depend on the
// other rows, and the merges run in fixed order, so a row's result depends
// only on its query, keys, limit and SP: not on the other rows of its block,
// the window size, the batch, or the merge path.  Keys past a row's limit
// contribute exact zeros.
#pragma once
#include "ptx.cuh"

namespace gs {

// K pages and V^T pages have rings of their own: a K page is done with S, a V^T
// page only a softmax and a P V later.  In one ring of 3 pairs a copy went out
// when P V of its predecessor ended and was wanted one page later (the MMA warp
// waited 610 of 1,700 cycles per page for it, 32 x U[1024, 6144] slots); here a
// K copy has 4 pages of lead and a V^T copy 3, in what two CTAs per SM can hold.
constexpr int kAttnKStages = 4, kAttnVStages = 3;
constexpr int kAttnPageBytes = 64 * 128;  // 64 x 64 fp16
constexpr int kAttnOnesBytes = 16 * 128;  // 16 rows of fp16 ones after each V^T page
constexpr int kAttnVStageBytes = kAttnPageBytes + kAttnOnesBytes;
constexpr int kAttnRow = 68;              // partial row: O[64], m, l, 2 pad (272 B)
constexpr int kAttnMaxRows = 128;         // rows of one query block (the MMA's M)
constexpr int kAttnMaxCluster = 16;       // items merged inside a cluster (16: non-portable size)
constexpr int kAttnSoftWarps = 4;         // one warp per TMEM lane quarter
constexpr int kAttnSoftThreads = kAttnSoftWarps * 32;
constexpr int kAttnThreads = kAttnSoftThreads + 64;   // + TMA warp, MMA warp
constexpr int kAttnTmaWarp = kAttnSoftWarps, kAttnMmaWarp = kAttnSoftWarps + 1;
constexpr int kAttnTmemCols = 256;        // S[2] at columns 0, 64; O at 128
constexpr int kAttnPtAhead = 64;         // page numbers an item reads up front
constexpr float kAttnRescale = 8.0f;      // log2 growth of the max that forces a rescale
constexpr int kAttnKRingBytes = kAttnKStages * kAttnPageBytes;
constexpr int kAttnRingBytes = kAttnKRingBytes + kAttnVStages * kAttnVStageBytes;
// Q [128][128 B] | P[2] [128][128 B] | K ring | V^T ring | barriers.  After the
// pages are done, Q and P hold the owner-grouped rows (cluster) and the rings
// the received rows.
constexpr int kAttnQOff = 0;
constexpr int kAttnPOff = kAttnMaxRows * 128;
constexpr int kAttnRingOff = kAttnPOff + 2 * kAttnMaxRows * 128;
constexpr int kAttnBarOff = kAttnRingOff + kAttnRingBytes;
constexpr int kAttnSmemBytes = 1024 + kAttnBarOff + 256 + kAttnMaxRows * 4 + kAttnPtAhead * 4;
constexpr int kAttnRowsFloats = (kAttnMaxRows + kAttnMaxCluster) * kAttnRow;
static_assert(kAttnRingOff >= kAttnRowsFloats * 4 && kAttnRingBytes >= kAttnRowsFloats * 4,
              "Q + P hold the owner-grouped rows, the ring the received rows");
// Items one merge through global scratch takes (an interface limit).
constexpr int kAttnMaxMergeItems = 54;

struct AttnArgs {
  const __half* q;            // [T, Hq, 64]
  const int32_t* lim;         // [T] inclusive key limit per query token
  __half* out;                // [T, Hq, 64]
  const int32_t* page_table;  // [slots, pt_stride]
  int pt_stride;
  const int32_t* blk_slot;    // [n_seq] page-table row per sequence, or null -> fixed_slot
  const int32_t* blk_active;  // [n_seq] nonzero = run, or null
  int fixed_slot;
  int T;                      // tokens
  int QB;                     // tokens per sequence window (prefill: per block)
  int QS, n_sub;              // tokens per query block; blocks per window
  int Hq, Hkv, G;
  int g_magic;                // ceil(2^16 / G): r / G = r * g_magic >> 16 for block rows r < 128
  long long kv_row_base;      // first KV-map row of this layer
  int rows_per_page;          // 2 * Hkv * 64
  int split_pages;            // SP: pages per item
  int max_items;              // items per (block, head) the grid covers
  int cluster;                // 1: attn_paged_kernel, a cluster of max_items (<= 16) CTAs; 0: attn_stream_kernel
  int early;                  // 1: the launch before this one does not write the descriptors or limits
  float* part;                // global merge: [n_blocks][Hkv][max_items] tiles of 128 * kAttnRow floats
  int* ticket;                // global merge: [n_blocks][Hkv], zero between launches
  int* err;
};

__host__ __device__ inline int attn_max_smem_bytes() { return kAttnSmemBytes; }

__device__ __forceinline__ uint32_t sw128(int row, int chunk) {
  return static_cast<uint32_t>(row * 128 + ((chunk ^ (row & 7)) << 4));
}

// 16 TMEM lanes x 64 (x8) or 8 (x1) fp32 columns, in the 16x256b fragment
// layout: thread t receives, for column group j (8 columns), r[4 j + 2 q + e] =
// lane t / 4 + 8 q, column 8 j + 2 (t mod 4) + e.  A row is spread over four
// neighbouring threads.
__device__ __forceinline__ void tmem_ld_16x256b_x8(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_16x256b_x1(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_st_16x256b_x1(uint32_t taddr, const uint32_t (&r)[4]) {
  asm volatile("tcgen05.st.sync.aligned.16x256b.x1.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr),
               "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3])
               : "memory");
}

__device__ __forceinline__ uint32_t tmem_ld1(uint32_t taddr) {
  uint32_t r;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr));
  return r;
}

// 2^x on the SFU (PTX ex2.approx.ftz.f32, one instruction): the P values are
// 2^(s - m) <= 2^8, and a result below the fp32 normal range is an fp16 zero.
__device__ __forceinline__ float ex2_sfu(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// max of three (PTX max.f32 with three sources, sm_100 and later)
__device__ __forceinline__ float fmax3(float x, float y, float z) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(x), "f"(y), "f"(z));
  return r;
}

// Barriers and buffers the softmax warps share with the MMA warp.
struct AttnSync {
  uint64_t *s_full, *s_free, *p_full;
  uint64_t* v_empty;   // [V stages] O += P V of the stage's page retired
  uint8_t* sP;         // [2][128][128 B]
  float* m_row;      // [128] per MMA row: the final running max
};

// MMA row (TMEM lane) -> block row, and back.
__device__ __forceinline__ int attn_block_row(int mrow) { return (mrow & 31) * 4 + (mrow >> 5); }

// Key limits of the rows a thread shares: set q (rows 8 q + lane / 4 of the
// quarter), -1 past the block's rows.
__device__ __forceinline__ void attn_row_limits(const AttnArgs& a, int warp, int R, int tok0,
                                                int (&lim)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int rr = (8 * q + ((threadIdx.x & 31) >> 2)) * 4 + warp;
    lim[q] = rr < R ? a.lim[tok0 + (rr * a.g_magic >> 16)] : -1;
  }
}

// This thread's 8 of the 1,024 16-byte pieces of the block's Q rows (MMA row i
// holds block row attn_block_row(i), zero past R), all loads in flight
// together; then into the swizzled Q tile (rows past the last set are not read).
__device__ __forceinline__ void attn_load_q(const AttnArgs& a, int h, int tok0, int R, uint4 (&v)[8]) {
  const int ch = threadIdx.x & 7, i0 = threadIdx.x >> 3;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int rr = attn_block_row(i0 + 16 * k);
    v[k] = make_uint4(0, 0, 0, 0);
    if (rr < R) {
      const int tt = rr * a.g_magic >> 16;
      const int hq = h * a.G + rr - tt * a.G;
      v[k] = *reinterpret_cast<const uint4*>(a.q + (static_cast<size_t>(tok0 + tt) * a.Hq + hq) * 64 + ch * 8);
    }
  }
}
__device__ __forceinline__ void attn_store_q(uint8_t* sQ, int R, const uint4 (&v)[8]) {
  const int ch = threadIdx.x & 7, i0 = threadIdx.x >> 3;
  const int lanes_used = ((R + 3) / 4 + 7) / 8 * 8;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int i = i0 + 16 * k;
    if ((i & 31) < lanes_used) *reinterpret_cast<uint4*>(sQ + sw128(i, ch)) = v[k];
  }
}

// Where the softmax warps' rings stand, kept from one item to the next.
struct AttnRings {
  RingPos s;   // S / P buffer of the next page
  RingPos v;   // V^T ring stage of the next page
};

// Online softmax over the item's pages for one warp and the rows of its lane
// quarter.  S comes from TMEM in the 16x256b layout, so a row is spread over
// four neighbouring threads and a set of 8 rows costs a thread 16 columns,
// whatever the number of rows in the block is: 34 rows (a 17-token window,
// GQA 2) cost 16 or 32 exponentials per thread and page.  Per page: S, mask and
// scale, the row's maximum (two shuffles); the row's running max m (log2 units)
// only moves when a page raises it by more than 2^8 (always on the first page,
// rarely after).  A rise rescales O and the row sum in O's column 64 (the
// previous O += P V must have retired); then P_j = exp2(s - m) as fp16 into the
// P tile.  No step of a page needs another warp: the warps meet only on the MMA
// warp's barriers.  Bound by the serial chain of a page (TMEM load, max,
// exponentials, P store, fence).
//
// The quarter's two 16-lane halves run through one rolled loop and the mask and
// the rescale are loops too: every CTA of a launch fetches this code again (the
// SM's instruction cache does not hold a kernel of 100 KB), and the four
// unrolled variants this replaces spent 10 k of a CTA's 34 k cycles on that.
// Waits are bounded; a warp whose wait ran out keeps arriving on the MMA
// warp's barriers to the last page.  Returns false if a wait ran out.
__device__ __forceinline__ bool attn_softmax(const AttnArgs& a, const AttnSync& y, uint32_t tmem,
                                             int warp, int nset, int np, int p_begin,
                                             const int (&lim)[4], AttnRings& rg) {
  const int lane = threadIdx.x & 31;
  const int quad = lane & 3;
  float m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
  int full_lim = 0x7FFFFFFF;   // every row of the warp sees the keys up to here
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (lim[q] >= 0) full_lim = min(full_lim, lim[q]);
  full_lim = __reduce_min_sync(0xFFFFFFFFu, full_lim);
  const uint32_t trow = tmem + (static_cast<uint32_t>(warp * 32) << 16);
  // row (warp * 32 + lane / 4) of the P tile; chunk j of row r sits at (j ^ (r & 7)) * 16
  const uint32_t p0 = smem_u32(y.sP) + (warp * 32 + (lane >> 2)) * 128 + ((lane >> 2) << 4) + 4 * quad;
  const uint32_t s_full0 = smem_u32(y.s_full), s_free0 = smem_u32(y.s_free), p_full0 = smem_u32(y.p_full);
  const float kScaleLog2 = 0.125f * 1.4426950408889634f;   // 1/sqrt(64) in log2 units
  bool ok = true;
  // waits are warp-uniform; after a failure the warp stops waiting
  auto wwait = [&](uint32_t bar, uint32_t parity) {
    if (ok) ok = __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, a.err)) != 0;
    return ok;
  };
  RingPos prev;          // V^T ring stage of page j - 1
  bool pv_seen = true;   // O += P V of page j - 1 is known to have retired
#pragma unroll 1
  for (int j = 0; j < np; ++j) {
    const int buf = rg.s.s;
    const bool have = wwait(s_full0 + 8 * buf, rg.s.ph);
    const int key0 = (p_begin + j) * 64;
    if (have) {
      tc_fence_after();
#pragma unroll 1
      for (int hf = 0; 2 * hf < nset; ++hf) {
        const bool two = 2 * hf + 1 < nset;   // the half's second set holds rows
        float mh[2] = {hf ? m[2] : m[0], hf ? m[3] : m[1]};
        const uint32_t half = static_cast<uint32_t>(16 * hf) << 16;
        // 1. S_j of the half; the buffer is free once every warp has read it
        uint32_t sr[32];
        tmem_ld_16x256b_x8(trow + half + buf * 64, sr);
        tmem_wait_ld();
        if (2 * hf + 2 >= nset) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(s_free0 + 8 * buf);
        }
        // 2. mask: keys past the row's limit (only on a window's last pages)
        if (key0 + 63 > full_lim) {
          const int l0 = hf ? lim[2] : lim[0], l1 = hf ? lim[3] : lim[1];
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const int key = key0 + 8 * (k >> 1) + 2 * quad + (k & 1);
            uint32_t& v0 = sr[4 * (k >> 1) + (k & 1)];
            uint32_t& v1 = sr[4 * (k >> 1) + 2 + (k & 1)];
            v0 = key <= l0 ? v0 : 0xFF800000u;
            v1 = key <= l1 ? v1 : 0xFF800000u;
          }
        }
        // 3. the rows' page max (of the unscaled scores; the scale is positive)
        //    over the four threads of a row; does any row rise by more than 2^8?
        float pm[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          auto S = [&](int k) { return __uint_as_float(sr[4 * (k >> 1) + 2 * q + (k & 1)]); };
          float t = fmax3(fmax3(S(0), S(1), S(2)), fmax3(S(3), S(4), S(5)), fmax3(S(6), S(7), S(8)));
          t = fmax3(t, fmax3(S(9), S(10), S(11)), fmax3(S(12), S(13), fmaxf(S(14), S(15))));
          t = fmaxf(t, __shfl_xor_sync(0xFFFFFFFFu, t, 1));
          t = fmaxf(t, __shfl_xor_sync(0xFFFFFFFFu, t, 2));
          pm[q] = t * kScaleLog2;
        }
        const bool rise0 = pm[0] > mh[0] + kAttnRescale;
        const bool rise1 = two && pm[1] > mh[1] + kAttnRescale;
        // 4. a rise rescales O and the row sum first.  tcgen05.ld / st are
        //    warp-collective: a half with any rising row rescales all its rows,
        //    the others by exactly 1.
        if (__any_sync(0xFFFFFFFFu, rise0 || rise1)) {
          const float al0 = !rise0 ? 1.f : (mh[0] == -INFINITY ? 0.f : exp2f(mh[0] - pm[0]));
          const float al1 = !rise1 ? 1.f : (mh[1] == -INFINITY ? 0.f : exp2f(mh[1] - pm[1]));
          if (rise0) mh[0] = pm[0];
          if (rise1) mh[1] = pm[1];
          if (hf) {
            m[2] = mh[0];
            m[3] = mh[1];
          } else {
            m[0] = mh[0];
            m[1] = mh[1];
          }
          if (!pv_seen) pv_seen = wwait(smem_u32(&y.v_empty[prev.s]), prev.ph);
          if (j > 0 && pv_seen) {
            tc_fence_after();
            const uint32_t o = trow + half + 128;
#pragma unroll 1
            for (int cg = 0; cg < 9; ++cg) {   // 8 columns each; the last: the row sums
              uint32_t v[4];
              tmem_ld_16x256b_x1(o + 8 * cg, v);
              tmem_wait_ld();
#pragma unroll
              for (int k = 0; k < 4; ++k)
                v[k] = __float_as_uint((k < 2 ? al0 : al1) * __uint_as_float(v[k]));
              tmem_st_16x256b_x1(o + 8 * cg, v);
            }
            tmem_wait_st();
          }
        }
        // 5. P_j = exp2(s - m) (fp16) into the rows of the P tile
        const uint32_t prow = p0 + buf * (kAttnMaxRows * 128) + hf * (16 * 128);
        auto put = [&](int q, float mq, uint32_t row) {
          const float sub = (mq == -INFINITY) ? 0.f : mq;
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) {
            const float x0 = ex2_sfu(fmaf(__uint_as_float(sr[4 * jj + 2 * q]), kScaleLog2, -sub));
            const float x1 = ex2_sfu(fmaf(__uint_as_float(sr[4 * jj + 2 * q + 1]), kScaleLog2, -sub));
            const __half2 hv = __floats2half2_rn(x0, x1);
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(row ^ (jj << 4)),
                         "r"(*reinterpret_cast<const uint32_t*>(&hv))
                         : "memory");
          }
        };
        put(0, mh[0], prow);
        if (two) put(1, mh[1], prow + 8 * 128);
      }
      fence_proxy_async_smem();
    }
    if ((!have || nset == 0) && lane == 0) mbar_arrive(s_free0 + 8 * buf);
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(p_full0 + 8 * buf);
    prev = rg.v;
    rg.v.next(kAttnVStages);
    rg.s.next(2);
    pv_seen = false;
  }
  if (quad == 0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) y.m_row[warp * 32 + 8 * q + (lane >> 2)] = m[q];
  }
  return ok;
}

__global__ void __launch_bounds__(kAttnThreads, 2)
    attn_paged_kernel(const __grid_constant__ CUtensorMap tmKV, const AttnArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0);   // warp-uniform
  const int lane = threadIdx.x & 31;
  constexpr int rows_alloc = kAttnMaxRows;
  uint8_t* sQ = smem + kAttnQOff;
  uint8_t* sP = smem + kAttnPOff;                        // [2][128][128 B]
  uint8_t* ring = smem + kAttnRingOff;                   // K pages
  uint8_t* vring = ring + kAttnKRingBytes;               // V^T pages, 16 rows of ones behind each
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kAttnBarOff);
  uint64_t* k_full = bars;                               // [K stages] TMA landed
  uint64_t* k_empty = k_full + kAttnKStages;             // [K stages] S of the page done
  uint64_t* v_full = k_empty + kAttnKStages;             // [V stages] TMA landed
  uint64_t* v_empty = v_full + kAttnVStages;             // [V stages] PV of the page done
  uint64_t* s_full = v_empty + kAttnVStages;             // [2] S in TMEM
  uint64_t* s_free = s_full + 2;                         // [2] S read by the softmax warps
  uint64_t* p_full = s_full + 4;                         // [2] P in smem (softmax warps' arrivals)
  uint64_t* mma_done = s_full + 6;                       // every MMA of this CTA retired
  uint64_t* recv_bar = s_full + 7;
  uint64_t* q_full = s_full + 8;                         // Q tile in smem (4 warp arrivals)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_full + 9);
  // [0] max limit, [1] last-item flag, [2] K and [3] V^T pages the MMA warp
  // took, [4] K and [5] V^T pages issued, [6] sequence active, [7] page-table row
  int* s_int = reinterpret_cast<int*>(s_full + 10);
  float* m_row = reinterpret_cast<float*>(s_int + 8);    // [128] running max per MMA row
  int* pt_s = reinterpret_cast<int*>(m_row + kAttnMaxRows);   // the item's first page numbers

  const int c = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const int seq = b / a.n_sub, sub = b % a.n_sub;
  // Before griddepcontrol.wait this kernel reads only what the kernel right
  // before it (the QKV GEMM, which writes q and the window's K/V) does not
  // write: the window descriptors (key limits, block slots), the page table,
  // and cache pages wholly before the current window.  Every early exit is
  // uniform across the CTA, and across the cluster before its barrier.
  const int tok0 = seq * a.QB + sub * a.QS;
  const int ntok = min(min(a.QS, a.QB - sub * a.QS), a.T - tok0);
  if (ntok <= 0) return;
  const int R = ntok * a.G;

  // One round of global latency: warp 0 reads the block's descriptors while
  // the others set up barriers, TMEM and the ones rows.
  if (warp == 0) {
    if (!a.early) pdl_wait();
    const int act = a.blk_active != nullptr ? a.blk_active[seq] : 1;
    const int sl = a.blk_slot ? a.blk_slot[seq] : a.fixed_slot;
    int lm[4];   // ntok <= 128
#pragma unroll
    for (int q = 0; q < 4; ++q) lm[q] = lane + 32 * q < ntok ? a.lim[tok0 + lane + 32 * q] : -1;
    const int mxl = __reduce_max_sync(0xFFFFFFFFu, max(max(lm[0], lm[1]), max(lm[2], lm[3])));
    if (lane == 0) {
      s_int[0] = mxl;
      s_int[6] = act;
      s_int[7] = sl;
    }
  } else if (warp == 1) {
    if (lane == 0) {
      for (int s = 0; s < 2 * (kAttnKStages + kAttnVStages); ++s) mbar_init(smem_u32(&bars[s]), 1);
      for (int i = 0; i < 2; ++i) {
        mbar_init(smem_u32(&s_full[i]), 1);
        mbar_init(smem_u32(&s_free[i]), kAttnSoftWarps);   // one arrival per softmax warp
        mbar_init(smem_u32(&p_full[i]), kAttnSoftWarps);
      }
      mbar_init(smem_u32(mma_done), 1);
      mbar_init(smem_u32(q_full), kAttnSoftWarps);
      mbar_init(smem_u32(recv_bar), 1);
      s_int[2] = s_int[3] = s_int[4] = s_int[5] = 0;
      fence_mbar_init();
    }
  } else if (warp < kAttnSoftWarps) {
    // the ones rows after every V^T page: O += P [V | 1] puts the row sum in O's column 64
    for (int i = threadIdx.x - 64; i < kAttnVStages * kAttnOnesBytes / 16; i += 64) {
      const int st = i / (kAttnOnesBytes / 16), off = i % (kAttnOnesBytes / 16);
      *reinterpret_cast<uint4*>(vring + st * kAttnVStageBytes + kAttnPageBytes + off * 16) =
          make_uint4(0x3C003C00u, 0x3C003C00u, 0x3C003C00u, 0x3C003C00u);
    }
    fence_proxy_async_smem();
  } else if (warp == kAttnTmaWarp) {
    if (lane == 0) tma_prefetch_desc(&tmKV);
  } else {
    tmem_alloc(smem_u32(tmem_slot), kAttnTmemCols);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int maxlim = s_int[0], slot = s_int[7];
  const int npages_blk = maxlim / 64 + 1;
  const int SP = a.split_pages;
  const int nitems = (npages_blk + SP - 1) / SP;
  const bool active = s_int[6] != 0;
  const bool bad = maxlim < 0 || npages_blk > a.pt_stride || slot < 0 || nitems > a.max_items ||
                   R > kAttnMaxRows;
  const bool in_cluster = nitems > 1;
  if (!active || bad || c >= nitems) {
    if (active && bad && threadIdx.x == 0) atomicExch(a.err, kErrBounds);
    // idle cluster member: counts in the cluster barrier, owns nothing
    if (active && !bad && in_cluster) cluster_arrive_release();
    if (warp == kAttnMmaWarp) tmem_dealloc(tmem, kAttnTmemCols);
    return;
  }
  if (in_cluster && threadIdx.x == 0) {
    // nitems sources, ceil(128 / nitems) rows each, arrive by bulk copy (after
    // the cluster barrier below)
    const int rpo = (rows_alloc + nitems - 1) / nitems;
    mbar_arrive_expect_tx(smem_u32(recv_bar), static_cast<uint32_t>(nitems * rpo * kAttnRow * 4));
  }

  const int p_begin = c * SP;
  const int np = min(npages_blk, p_begin + SP) - p_begin;
  const int32_t* pt = a.page_table + static_cast<size_t>(slot) * a.pt_stride;
  bool ok = true;
  if (warp == kAttnTmaWarp) {
    // ---- TMA producer: K and V^T pages of the item, in order.  The first page
    // numbers come in one coalesced read; the rest are read a page ahead.
    for (int i = lane; i < min(np, kAttnPtAhead); i += 32) pt_s[i] = pt[p_begin + i];
    __syncwarp();
    if (elect_one()) {
      // pages wholly before the window: the limit of the WINDOW's first token (n or
      // n + 1); a later sub-block's own limits reach into slots that the kernel
      // right before this one is still writing
      const int safe_pages = a.blk_slot ? a.lim[seq * a.QB] / 64 : 0;
      const uint64_t pol = l2_policy_evict_first();
      RingPos rk, rv;
      const uint32_t k_full0 = smem_u32(k_full), k_empty0 = smem_u32(k_empty);
      const uint32_t v_full0 = smem_u32(v_full), v_empty0 = smem_u32(v_empty);
      const uint32_t k0 = smem_u32(ring), v0 = smem_u32(vring);
      int ahead = np > kAttnPtAhead ? pt[p_begin + kAttnPtAhead] : 0;
      int vrow = 0;   // pool row of the page whose V^T copy is next
      auto issue_k = [&](int i) {   // returns the page's V^T row
        int phys = i < kAttnPtAhead ? pt_s[i] : ahead;
        if (i >= kAttnPtAhead && i + 1 < np) ahead = pt[p_begin + i + 1];
        if (phys < 0) {  // unmapped page: the TMA box lands out of bounds and reads zeros
          atomicExch(a.err, kErrBounds);
          phys = 0x3FFFFFFF / a.rows_per_page;
        }
        const int row = static_cast<int>(a.kv_row_base + static_cast<long long>(phys) * a.rows_per_page);
        const uint32_t fb = k_full0 + 8 * rk.s;
        mbar_arrive_expect_tx(fb, kAttnPageBytes);
        tma_load_2d(k0 + rk.s * kAttnPageBytes, &tmKV, 0, row + h * 64, fb, pol);
        rk.next(kAttnKStages);
        s_int[4] = i + 1;
        return row + (a.Hkv + h) * 64;
      };
      auto issue_v = [&](int i, int row) {
        const uint32_t fb = v_full0 + 8 * rv.s;
        mbar_arrive_expect_tx(fb, kAttnPageBytes);   // the ones rows stay
        tma_load_2d(v0 + rv.s * kAttnVStageBytes, &tmKV, 0, row, fb, pol);
        rv.next(kAttnVStages);
        s_int[5] = i + 1;
      };
      // K of page i, then V^T of page i - 1: S runs a page ahead of P V
      int i = 0;
      const int npre = min(np, min(safe_pages - p_begin, kAttnVStages));
#pragma unroll 1
      for (; i < npre; ++i) {
        if (i > 0) issue_v(i - 1, vrow);
        vrow = issue_k(i);
      }
      pdl_wait();
      pdl_trigger();
#pragma unroll 1
      for (; i <= np && ok; ++i) {
        int next_vrow = 0;
        if (i < np) {
          if (i >= kAttnKStages && !mbar_wait(k_empty0 + 8 * rk.s, rk.ph ^ 1, a.err)) {
            ok = false;
            break;
          }
          next_vrow = issue_k(i);
        }
        if (i > 0) {
          if (i > kAttnVStages && !mbar_wait(v_empty0 + 8 * rv.s, rv.ph ^ 1, a.err)) {
            ok = false;
            break;
          }
          issue_v(i - 1, vrow);
        }
        vrow = next_vrow;
      }
    } else {
      pdl_wait();
      pdl_trigger();
    }
  } else if (warp == kAttnMmaWarp) {
    // ---- MMA issuer: S one page ahead of the softmax, O += P V after each P
    pdl_wait();
    pdl_trigger();
    if (elect_one()) {
      constexpr uint32_t idesc = umma_idesc_f16(128, 64);
      constexpr uint32_t idesc_pv = umma_idesc_f16(128, 80);   // V^T page and its 16 ones rows
      const uint64_t qdesc = umma_desc_sw128(smem_u32(sQ));
      const uint64_t pdesc0 = umma_desc_sw128(smem_u32(sP));
      const uint64_t kdesc0 = umma_desc_sw128(smem_u32(ring));
      const uint64_t vdesc0 = umma_desc_sw128(smem_u32(vring));
      const uint32_t k_full0 = smem_u32(k_full), k_empty0 = smem_u32(k_empty);
      const uint32_t v_full0 = smem_u32(v_full), v_empty0 = smem_u32(v_empty);
      const uint32_t s_full0 = smem_u32(s_full), s_free0 = smem_u32(s_free), p_full0 = smem_u32(p_full);
      RingPos rk, rv;   // ring stages of the next S and the next PV
      auto issue_s = [&](int j) -> bool {
        const int buf = j & 1;
        if (!mbar_wait(k_full0 + 8 * rk.s, rk.ph, a.err)) return false;
        s_int[2] = j + 1;
        if (j >= 2 && !mbar_wait(s_free0 + 8 * buf, ((j >> 1) + 1) & 1, a.err)) return false;
        tc_fence_after();
        const uint64_t kdesc = kdesc0 + rk.s * (kAttnPageBytes >> 4);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          umma_f16(tmem + buf * 64, qdesc + 2 * k, kdesc + 2 * k, idesc, k > 0 ? 1u : 0u);
        umma_commit(s_full0 + 8 * buf);
        umma_commit(k_empty0 + 8 * rk.s);
        rk.next(kAttnKStages);
        return true;
      };
      if (!mbar_wait(smem_u32(q_full), 0, a.err)) ok = false;   // Q tile written
      if (ok) ok = issue_s(0);
#pragma unroll 1
      for (int j = 0; j < np && ok; ++j) {
        if (j + 1 < np && !(ok = issue_s(j + 1))) break;
        const int buf = j & 1;
        if (!mbar_wait(v_full0 + 8 * rv.s, rv.ph, a.err)) {
          ok = false;
          break;
        }
        s_int[3] = j + 1;
        if (!mbar_wait(p_full0 + 8 * buf, (j >> 1) & 1, a.err)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t pdesc = pdesc0 + buf * (kAttnMaxRows * 128 >> 4);
        const uint64_t vdesc = vdesc0 + rv.s * (kAttnVStageBytes >> 4);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          umma_f16(tmem + 128, pdesc + 2 * k, vdesc + 2 * k, idesc_pv, (j > 0 || k > 0) ? 1u : 0u);
        umma_commit(v_empty0 + 8 * rv.s);
        rv.next(kAttnVStages);
      }
      umma_commit(smem_u32(mma_done));   // retires once every MMA above has
    }
  } else {
    // ---- softmax warps: Q rows -> swizzled smem (MMA row i holds block row
    // attn_block_row(i), zero past R; rows past the last set are not read)
    const int rows_w = warp < R ? (R - warp + 3) / 4 : 0;   // rows in this warp's quarter
    pdl_wait();
    pdl_trigger();
    uint4 v[8];
    attn_load_q(a, h, tok0, R, v);
    attn_store_q(sQ, R, v);
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(q_full));
    AttnSync y{s_full, s_free, p_full, v_empty, sP, m_row};
    int lim[4];
    attn_row_limits(a, warp, R, tok0, lim);
    AttnRings rg;
    ok = attn_softmax(a, y, tmem, warp, (rows_w + 7) / 8, np, p_begin, lim, rg);
  }

  // every MMA retired and every TMA copy landed before TMEM and the ring are reused
  if (warp == kAttnTmaWarp) {
    __syncwarp();   // the elected thread's page counts are written
  } else {
    mbar_wait(smem_u32(mma_done), 0, a.err);
  }
  const bool all_ok = __syncthreads_and(ok);
  if (!all_ok) {   // a wait ran out: pages that were issued and not taken may still be landing
    if (threadIdx.x == 0) {
#pragma unroll 1
      for (int i = s_int[2]; i < s_int[4]; ++i)
        mbar_wait(smem_u32(&k_full[i % kAttnKStages]), (i / kAttnKStages) & 1, a.err);
#pragma unroll 1
      for (int i = s_int[3]; i < s_int[5]; ++i)
        mbar_wait(smem_u32(&v_full[i % kAttnVStages]), (i / kAttnVStages) & 1, a.err);
    }
    __syncthreads();
  }
  // the row's O and its sum (O's column 64) from TMEM (rows < R)
  const int r = warp < kAttnSoftWarps ? attn_block_row(threadIdx.x) : kAttnMaxRows;   // block row
  const bool row_thread = r < R;
  float o[64];
  float m = -INFINITY, l = 0.f;   // the row's running max (log2 units) and sum
  if (warp < 4) {
    tc_fence_after();
    uint32_t o0[32], o1[32];
    tmem_ld32_nowait(tmem + (static_cast<uint32_t>(warp * 32) << 16) + 128, o0);
    tmem_ld32_nowait(tmem + (static_cast<uint32_t>(warp * 32) << 16) + 128 + 32, o1);
    const uint32_t l1 = tmem_ld1(tmem + (static_cast<uint32_t>(warp * 32) << 16) + 192);
    tmem_wait_ld();
    m = m_row[threadIdx.x];
    l = __uint_as_float(l1);
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      o[k] = __uint_as_float(o0[k]);
      o[32 + k] = __uint_as_float(o1[k]);
    }
  }
  tc_fence_before();

  // (the MMA warp frees TMEM behind the barrier that follows the row stores)
  auto free_tmem = [&] {
    if (warp == kAttnMmaWarp) {
      tc_fence_after();
      tmem_dealloc(tmem, kAttnTmemCols);
    }
  };
  if (nitems == 1) {   // the block's only item: its rows are final
    if (row_thread && all_ok) {
      const float inv = 1.0f / l;
      const int tt = r * a.g_magic >> 16;
      const int t = tok0 + tt;
      const int hq = h * a.G + r - tt * a.G;
      __half* dst = a.out + (static_cast<size_t>(t) * a.Hq + hq) * 64;
#pragma unroll
      for (int cch = 0; cch < 8; ++cch) {
        uint32_t w4[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          __half2 hv = __floats2half2_rn(o[8 * cch + 2 * e] * inv, o[8 * cch + 2 * e + 1] * inv);
          w4[e] = *reinterpret_cast<uint32_t*>(&hv);
        }
        *reinterpret_cast<uint4*>(dst + 8 * cch) = make_uint4(w4[0], w4[1], w4[2], w4[3]);
      }
    }
    __syncthreads();
    free_tmem();
    return;
  }

  // this thread's row (O, m, l) -> a [kAttnRow] slot
  auto put_row = [&](float* dst) {
#pragma unroll
    for (int k = 0; k < 64; k += 4)
      *reinterpret_cast<float4*>(dst + k) = make_float4(o[k], o[k + 1], o[k + 2], o[k + 3]);
    *reinterpret_cast<float2*>(dst + 64) = make_float2(m, l);
  };

  // ---- items -> owners: CTA c of the cluster owns rows c, c + nitems, ...
  // Outgoing rows [owner][slot][kAttnRow] over Q and P, received rows
  // recv[it][k] (row c + k * nitems of item `it`) in the rings.
  float* stage = reinterpret_cast<float*>(sQ);
  float* recv = reinterpret_cast<float*>(ring);
  const int rpo = (rows_alloc + nitems - 1) / nitems;   // rows per owner
  const int blk_floats = rpo * kAttnRow;
  if (row_thread)
    put_row(stage + static_cast<size_t>(r % nitems) * blk_floats + (r / nitems) * kAttnRow);
  fence_proxy_async_smem();
  __syncthreads();
  free_tmem();
  cluster_arrive_release();
  cluster_wait();   // every CTA of the cluster is done with its pages: receive buffers idle
  if (threadIdx.x == 0) {
    const uint32_t bytes = static_cast<uint32_t>(blk_floats * 4);
    const uint32_t dst_local = smem_u32(recv) + static_cast<uint32_t>(c) * bytes;
#pragma unroll 1
    for (int q = 0; q < nitems; ++q)
      bulk_copy_to_peer(cluster_map(dst_local, static_cast<uint32_t>(q)),
                        smem_u32(stage) + static_cast<uint32_t>(q) * bytes, bytes,
                        cluster_map(smem_u32(recv_bar), static_cast<uint32_t>(q)));
    bulk_commit();
  }
  const bool got = mbar_wait(smem_u32(recv_bar), 0, a.err);
  const int my_rows = (R - c + nitems - 1) / nitems;

  // ---- merge of items 0..nitems-1 in order for the owned rows: one thread per
  //      (row, 4 dims); M = max m_i, w_i = 2^(m_i - M), L = sum w_i l_i,
  //      O = sum (w_i / L) O_i
#pragma unroll 1
  for (int idx = threadIdx.x; idx < my_rows * 16; idx += blockDim.x) {
    const int k = idx >> 4, d4 = (idx & 15) * 4;
    const float* row = recv + static_cast<size_t>(k) * kAttnRow;
    float M = -INFINITY, L = 0.f;
#pragma unroll 4
    for (int it = 0; it < nitems; ++it) M = fmaxf(M, row[it * blk_floats + 64]);
#pragma unroll 4
    for (int it = 0; it < nitems; ++it) {
      const float2 ml = *reinterpret_cast<const float2*>(row + it * blk_floats + 64);
      L += (ml.x == -INFINITY ? 0.f : exp2f(ml.x - M)) * ml.y;
    }
    const float inv = 1.0f / L;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int it = 0; it < nitems; ++it) {
      const float mi = row[it * blk_floats + 64];
      const float4 v = *reinterpret_cast<const float4*>(row + it * blk_floats + d4);
      const float w = (mi == -INFINITY ? 0.f : exp2f(mi - M)) * inv;
      acc.x += w * v.x;
      acc.y += w * v.y;
      acc.z += w * v.z;
      acc.w += w * v.w;
    }
    if (all_ok && got) {
      const int rr = c + k * nitems;
      const int tt = rr * a.g_magic >> 16;
      const int hq = h * a.G + rr - tt * a.G;
      __half* dst = a.out + (static_cast<size_t>(tok0 + tt) * a.Hq + hq) * 64 + d4;
      *reinterpret_cast<__half2*>(dst) = __floats2half2_rn(acc.x, acc.y);
      *reinterpret_cast<__half2*>(dst + 2) = __floats2half2_rn(acc.z, acc.w);
    }
  }
  if (threadIdx.x == 0) bulk_wait_read_all();   // our outgoing rows have left
}

}  // namespace gs
