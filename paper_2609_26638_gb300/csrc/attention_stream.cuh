// attention_stream.cuh -- the paged attention of attention.cuh for launches
// larger than about one wave of CTAs: persistent CTAs, two per SM, each taking
// one work item (item, KV head, query block) after another.
//
// The grid has a CTA per work item, items slowest (the ones past a short
// sequence's end come last); a running CTA takes over CTAs that have not started
// (cluster launch control), so the items of long and short sequences spread by
// themselves.  The producer warp fetches the next item's descriptors
// and streams its pages while the softmax warps still work on the last one, and
// it drops the CTAs whose item lies past the sequence's end: with a CTA per
// item, each paid 1.5 us of start-up, 0.9 us for Q and 2.5-3 us for its rows and
// ticket around 8 us of pages (13 pages of a 17-token window, 1.5 of 2 CTAs
// resident).  With the same page loop, 64 sequences of 8192 keys took 227 us with
// a CTA per item and 207 here, a prefill chunk of 1024 tokens 85.5 and 78, 32
// sequences of 1-6 k keys 80 and 81; with the merges' loads in flight together
// (attn_merge_rows) 194, 57.5 and 69.  The arithmetic and its order are
// attention.cuh's.
//
// Warps 0-3: softmax, the item's rows to global scratch, and merges; 4: producer
// (scheduling, descriptors, page copies, tickets); 5: MMA issue.  An item's rows
// are posted to the producer, which orders them before the (block, head)'s
// counter once the next item's copies are out; the answer -- this was the last
// item, merge -- is taken up after the next item's rows, so nobody waits for the
// fence and the atomic.
// The roles meet on mbarriers only: a wait that runs out ends its role, and the
// others' waits run out in turn.
#pragma once
#include "attention.cuh"

namespace gs {

// barriers and slots behind the rings: 31 barriers, the TMEM address, two work
// descriptors of 8 ints, the scheduler's answer, the ticket's answer
constexpr int kAttnStreamTail = 512;
constexpr int kAttnStreamSmem = 1024 + kAttnBarOff + kAttnStreamTail + kAttnMaxRows * 4 + kAttnPtAhead * 4;
static_assert(2 * (kAttnStreamSmem + 1024) <= 228 * 1024, "two CTAs per SM");

// An item's rows in global scratch: O [128][64], then (m, l) [128] -- whole 128-byte
// lines of O, and one line of (m, l) for 16 rows, where the merge reads them.
constexpr int kAttnTileMl = kAttnMaxRows * 64;
static_assert(kAttnTileMl + 2 * kAttnMaxRows <= kAttnMaxRows * kAttnRow, "the tile holds rows and (m, l)");

struct AttnWork {
  int np, p_begin, nitems, tok0, R, b, h, c;   // np == 0: no more work
};

// Merge of the items of a (block, head) by the softmax warps: M = max m_i,
// w_i = 2^(m_i - M), L = sum w_i l_i in item order, O = sum (w_i / L) O_i in item
// order.  First one thread per row leaves the coefficients w_i / L in `coef`
// [item][row] (over the idle P tiles), then a thread takes (row, 4 dims) units,
// two at a time: the rows come from L2, so loads in flight decide, and a launch
// ends with merges that nothing overlaps (two per CTA at worst).  The loads are
// unconditional and stand before a __syncwarp: with a condition on each, the
// compiler put every load beside its use, eight round trips in a row.  A merge of
// 98 rows of 8 items took 16.6 us so, 5.8 now; of 34 rows 7.1 and 3.6; of 10 rows
// of 27 items 12.2 (four loads of (m, l) at a time) and 6.5.  Launches: 10 windows
// of 49 tokens at 6000 slots 90.5 us so, 61.7 now (73 with a CTA per item), one
// window of 5 tokens at 8000 slots in 26 items 25.3 and 19.5 (21.4).
// `bar` completes two phases per merge: coefficients written, and read (the P
// tiles are the softmax's again).  False if a wait ran out.
__device__ __forceinline__ bool attn_merge_rows(const float* part, float* coef, __half* out, uint64_t* bar,
                                             int nitems, int R, int tok0, int h, int Hq, int G,
                                             int g_magic, int* err) {
  constexpr int kUnits = 2;
  const size_t step = static_cast<size_t>(kAttnMaxRows) * kAttnRow;   // item to item
  const int r = min(static_cast<int>(threadIdx.x), R - 1);
  const bool own = threadIdx.x < R;
  const float* row = part + kAttnTileMl + 2 * r;
  float* cf = coef + r;
  float M = -INFINITY, L = 0.f;
  if (nitems <= 8) {
    if (own) {
      float2 ml[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        ml[u] = u < nitems ? __ldcg(reinterpret_cast<const float2*>(row + u * step))
                           : make_float2(-INFINITY, 0.f);
#pragma unroll
      for (int u = 0; u < 8; ++u) M = fmaxf(M, ml[u].x);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (u < nitems) {
          ml[u].x = ml[u].x == -INFINITY ? 0.f : exp2f(ml[u].x - M);
          L += ml[u].x * ml[u].y;
        }
      const float inv = 1.0f / L;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (u < nitems) cf[u * kAttnMaxRows] = ml[u].x * inv;
    }
  } else if (static_cast<int>(threadIdx.x & ~31u) < R) {   // (warp-uniform)
    // sixteen loads in flight: the maxima, kept in the coefficients' places, then
    // the sums
#pragma unroll 1
    for (int it0 = 0; it0 < nitems; it0 += 16) {
      float v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = __ldcg(row + min(it0 + u, nitems - 1) * step);
      __syncwarp();
#pragma unroll
      for (int u = 0; u < 16; ++u) M = fmaxf(M, v[u]);   // (a repeated item changes no maximum)
#pragma unroll
      for (int u = 0; u < 16; ++u)
        if (own && it0 + u < nitems) cf[(it0 + u) * kAttnMaxRows] = v[u];
    }
#pragma unroll 1
    for (int it0 = 0; it0 < nitems; it0 += 16) {
      float v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = __ldcg(row + 1 + min(it0 + u, nitems - 1) * step);
      __syncwarp();
#pragma unroll
      for (int u = 0; u < 16; ++u)
        if (own && it0 + u < nitems) {
          float* c = cf + (it0 + u) * kAttnMaxRows;
          const float w = *c == -INFINITY ? 0.f : exp2f(*c - M);
          *c = w;
          L += w * v[u];
        }
    }
    const float inv = 1.0f / L;
    if (own) {
#pragma unroll 4
      for (int it = 0; it < nitems; ++it) cf[it * kAttnMaxRows] *= inv;
    }
  }
  auto meet = [&](uint32_t parity) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(smem_u32(bar));
    return __all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(bar), parity, err)) != 0;
  };
  if (!meet(0)) return false;
#pragma unroll 1
  for (int base = threadIdx.x & ~31; base < R * 16; base += kUnits * kAttnSoftThreads) {   // (warp-uniform)
    const int idx = base + (threadIdx.x & 31);
    float4 acc[kUnits];
    const float* src[kUnits];
    const float* w_of[kUnits];
#pragma unroll
    for (int q = 0; q < kUnits; ++q) {
      const int i = min(idx + q * kAttnSoftThreads, R * 16 - 1);
      acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
      src[q] = part + i * 4;
      w_of[q] = coef + (i >> 4);
    }
#pragma unroll 1
    for (int it0 = 0; it0 < nitems; it0 += 8) {
      float4 v[kUnits][8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int it = min(it0 + u, nitems - 1);
#pragma unroll
        for (int q = 0; q < kUnits; ++q)
          v[q][u] = __ldcg(reinterpret_cast<const float4*>(src[q] + it * step));
      }
      __syncwarp();   // the loads go out before the first one is used
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const bool live = it0 + u < nitems;
        const int it = min(it0 + u, nitems - 1);
#pragma unroll
        for (int q = 0; q < kUnits; ++q) {
          const float w = w_of[q][it * kAttnMaxRows];
          acc[q].x = live ? acc[q].x + w * v[q][u].x : acc[q].x;
          acc[q].y = live ? acc[q].y + w * v[q][u].y : acc[q].y;
          acc[q].z = live ? acc[q].z + w * v[q][u].z : acc[q].z;
          acc[q].w = live ? acc[q].w + w * v[q][u].w : acc[q].w;
        }
      }
    }
#pragma unroll
    for (int q = 0; q < kUnits; ++q) {
      const int i = idx + q * kAttnSoftThreads;
      if (i >= R * 16) break;
      const int tt = (i >> 4) * g_magic >> 16;
      const int hq = h * G + (i >> 4) - tt * G;
      __half* dst = out + (static_cast<size_t>(tok0 + tt) * Hq + hq) * 64 + (i & 15) * 4;
      *reinterpret_cast<__half2*>(dst) = __floats2half2_rn(acc[q].x, acc[q].y);
      *reinterpret_cast<__half2*>(dst + 2) = __floats2half2_rn(acc[q].z, acc[q].w);
    }
  }
  return meet(1);
}
static_assert(kAttnMaxMergeItems * kAttnMaxRows * 4 <= 2 * kAttnMaxRows * 128, "coefficients fit the P tiles");

__global__ void __launch_bounds__(kAttnThreads, 2)
    attn_stream_kernel(const __grid_constant__ CUtensorMap tmKV, const AttnArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0);   // warp-uniform
  const int lane = threadIdx.x & 31;
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
  uint64_t* q_full = s_full + 6;                         // the item's Q tile in smem
  uint64_t* o_full = s_full + 7;                         // the item's O complete
  uint64_t* o_free = s_full + 8;                         // O read by the softmax warps
  uint64_t* work_full = s_full + 9;                      // [2] work descriptor written
  uint64_t* work_free = s_full + 11;                     // [2] the item's rows are out, the MMA warp has read it
  uint64_t* clc_bar = s_full + 13;                       // the scheduler's answer
  uint64_t* rows_full = s_full + 14;                     // the item's rows are in global scratch
  uint64_t* tick_full = s_full + 15;                     // the ticket's answer
  uint64_t* merge_bar = s_full + 16;                     // a merge's coefficients are written, then read
  constexpr int kBars = 2 * (kAttnKStages + kAttnVStages) + 17;
  static_assert(kBars * 8 <= 256 && 256 + 64 + 16 + 16 <= kAttnStreamTail, "tail layout");
  uint32_t* clc_slot = reinterpret_cast<uint32_t*>(smem + kAttnBarOff + 256);        // 16 bytes
  AttnWork* work = reinterpret_cast<AttnWork*>(smem + kAttnBarOff + 272);            // [2]
  volatile int* tick = reinterpret_cast<volatile int*>(smem + kAttnBarOff + 336);    // last item?
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kAttnBarOff + 340);
  float* m_row = reinterpret_cast<float*>(smem + kAttnBarOff + kAttnStreamTail);     // [128]
  int* pt_s = reinterpret_cast<int*>(m_row + kAttnMaxRows);   // the item's first page numbers

  if (warp == 0) {
    if (lane == 0) {
#pragma unroll 1
      for (int i = 0; i < kBars; ++i) {
        uint64_t* bar = bars + i;
        const int n = bar >= s_free && bar < q_full + 1 ? kAttnSoftWarps
                      : (bar == o_free || bar == rows_full || bar == merge_bar) ? kAttnSoftWarps
                      : (bar == work_free || bar == work_free + 1) ? kAttnSoftWarps + 1 : 1;
        mbar_init(smem_u32(bar), n);
      }
      fence_mbar_init();
    }
  } else if (warp < kAttnSoftWarps) {
    // the ones rows after every V^T page: O += P [V | 1] puts the row sum in O's column 64
    for (int i = threadIdx.x - 32; i < kAttnVStages * kAttnOnesBytes / 16; i += 96) {
      const int st = i / (kAttnOnesBytes / 16), off = i % (kAttnOnesBytes / 16);
      *reinterpret_cast<uint4*>(vring + st * kAttnVStageBytes + kAttnPageBytes + off * 16) =
          make_uint4(0x3C003C00u, 0x3C003C00u, 0x3C003C00u, 0x3C003C00u);
    }
    fence_proxy_async_smem();
  } else if (warp == kAttnTmaWarp) {
    if (lane == 0) tma_prefetch_desc(&tmKV);
  } else if (warp == kAttnMmaWarp) {
    tmem_alloc(smem_u32(tmem_slot), kAttnTmemCols);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == kAttnTmaWarp) {
    // ---- producer.  While an item's pages go out it takes the last item's
    // ticket (after five: the softmax warps have begun this one) and asks for the
    // next CTA (three pages before the end); the softmax warps still have the
    // rings' pages when it has looked at the answer.  Asking earlier let a third
    // of the CTAs hold two items the others could have begun (64 x 8192 slots,
    // K 32, 8 sequences: half the CTAs done at 40 us, the last at 69).
    RingPos ws;
    uint32_t clc_ph = 0, rows_ph = 0;
    int issued = 0;   // pages so far: the rings' positions
    int published = 0, tickets = 0;
    bool ok = true, first = true, asked = false, left = true, own = true;
    const uint64_t pol = l2_policy_evict_first();
    const uint32_t k_full0 = smem_u32(k_full), k_empty0 = smem_u32(k_empty);
    const uint32_t v_full0 = smem_u32(v_full), v_empty0 = smem_u32(v_empty);
    const uint32_t k0 = smem_u32(ring), v0 = smem_u32(vring);
    // the item being fetched (np == 0: none left)
    AttnWork nw;
    const int32_t* npt = nullptr;   // its page-table entries
    int nsafe = 0, np0 = 0, np1 = 0;   // wholly committed pages; page numbers lane, lane + 32

    // Look at CTA (c, h, b): its item's descriptor into nw (np = 0: no item).
    // Until griddepcontrol.wait this kernel reads only what the kernel right
    // before it (the QKV GEMM) does not write: key limits, block slots, the page
    // table, and cache pages wholly before the current window.
    auto look = [&](int c, int h, int b) {
      const int seq = b / a.n_sub, sub = b - seq * a.n_sub;
      const int tok0 = seq * a.QB + sub * a.QS;
      const int ntok = min(min(a.QS, a.QB - sub * a.QS), a.T - tok0);
      nw.np = 0;
      if (ntok <= 0) return;
      const int act = a.blk_active != nullptr ? a.blk_active[seq] : 1;
      const int slot = a.blk_slot ? a.blk_slot[seq] : a.fixed_slot;
      int lm[4];   // ntok <= 128
#pragma unroll
      for (int q = 0; q < 4; ++q) lm[q] = lane + 32 * q < ntok ? a.lim[tok0 + lane + 32 * q] : -1;
      // pages wholly before the window, from the window's first token (a later
      // sub-block's own limits reach into the window)
      nsafe = a.blk_slot ? a.lim[seq * a.QB] / 64 : 0;
      const int maxlim = __reduce_max_sync(0xFFFFFFFFu, max(max(lm[0], lm[1]), max(lm[2], lm[3])));
      const int npages = maxlim / 64 + 1;
      const int nitems = (npages + a.split_pages - 1) / a.split_pages;
      const bool bad = maxlim < 0 || npages > a.pt_stride || slot < 0 || nitems > a.max_items ||
                       ntok * a.G > kAttnMaxRows;
      if (act != 0 && bad && lane == 0) atomicExch(a.err, kErrBounds);
      if (act == 0 || bad || c >= nitems) return;
      const int p_begin = c * a.split_pages;
      nw = AttnWork{min(npages, p_begin + a.split_pages) - p_begin, p_begin, nitems, tok0, ntok * a.G, b, h, c};
      npt = a.page_table + static_cast<size_t>(slot) * a.pt_stride + p_begin;
      np0 = lane < nw.np ? npt[lane] : 0;
      np1 = lane + 32 < nw.np ? npt[lane + 32] : 0;
    };
    auto ask = [&] {
      if (elect_one()) {
        mbar_arrive_expect_tx(smem_u32(clc_bar), 16);
        clc_try_cancel(smem_u32(clc_slot), smem_u32(clc_bar));
      }
      asked = true;
    };
    // The next CTA that has an item -- first this one -- into nw; false if a wait
    // ran out.
    auto fetch = [&]() -> bool {
      nw.np = 0;
      int h = blockIdx.x, b = blockIdx.y, c = blockIdx.z;
#pragma unroll 1
      while (left && nw.np == 0) {
        if (!own) {
          if (!asked) ask();
          if (!__all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(clc_bar), clc_ph, a.err))) return false;
          clc_ph ^= 1;
          asked = false;
          left = clc_answer(smem_u32(clc_slot), &h, &b, &c);
          fence_proxy_async_smem();   // read before the next answer is written
          __syncwarp();
          if (!left) break;
        }
        own = false;
        look(c, h, b);
      }
      return true;
    };
    // The ticket of item number `tickets`, whose descriptor is in its slot: its
    // rows, then the (block, head)'s counter.
    auto ticket = [&]() -> bool {
      bool good = true;
      if (lane == 0) {
        const AttnWork t = work[tickets & 1];
        if (t.nitems > 1) {
          good = mbar_wait(smem_u32(rows_full), rows_ph, a.err);
          rows_ph ^= 1;
          if (good) {
            int* cnt = a.ticket + static_cast<size_t>(t.b) * a.Hkv + t.h;
            __threadfence();
            const bool last = atomicAdd(cnt, 1) == t.nitems - 1;
            __threadfence();
            if (last) *cnt = 0;   // every item of this launch has arrived
            *tick = last ? 1 : 0;
            mbar_arrive(smem_u32(tick_full));
          }
        }
      }
      ++tickets;
      return __all_sync(0xFFFFFFFFu, good) != 0;
    };
    // Publish nw (or the end) in the next slot.
    auto publish = [&]() -> bool {
      if (!__all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(work_free) + 8 * ws.s, ws.ph ^ 1, a.err))) return false;
      pt_s[lane] = np0;        // kAttnPtAhead == 64 page numbers up front
      pt_s[lane + 32] = np1;
      if (lane == 0) {
        work[ws.s] = nw;
        mbar_arrive(smem_u32(work_full) + 8 * ws.s);
      }
      __syncwarp();
      ws.next(2);
      ++published;
      return true;
    };
    // Pages [i0, i1) of the item published last (K of page i, then V^T of page
    // i - 1: S runs a page ahead of P V; i == np: V^T of the last).
    auto stream = [&](int i0, int i1, int np, int p_begin, int safe_pages, int h, const int32_t* pt) -> bool {
      bool good = true;
      if (elect_one()) {
        RingPos rk, rv;
        const int kn = issued + i0, vn = issued + (i0 > 0 ? i0 - 1 : 0);
        rk.s = kn % kAttnKStages;
        rk.ph = (kn / kAttnKStages) & 1;
        rv.s = vn % kAttnVStages;
        rv.ph = (vn / kAttnVStages) & 1;
        auto row_of = [&](int i) {
          int phys = i < kAttnPtAhead ? pt_s[i] : pt[i];
          if (phys < 0) {  // unmapped page: the TMA box lands out of bounds and reads zeros
            atomicExch(a.err, kErrBounds);
            phys = 0x3FFFFFFF / a.rows_per_page;
          }
          return static_cast<int>(a.kv_row_base + static_cast<long long>(phys) * a.rows_per_page);
        };
        const int npre = min(np, min(safe_pages - p_begin, kAttnVStages));
        int vrow = i0 > 0 ? row_of(i0 - 1) : 0;   // the page whose V^T copy is next
#pragma unroll 1
        for (int i = i0; i < i1; ++i) {
          if (first && i >= npre) {
            pdl_wait();
            pdl_trigger();
            first = false;
          }
          int row = 0;
          if (i < np) {
            row = row_of(i);
            if (!(good = mbar_wait(k_empty0 + 8 * rk.s, rk.ph ^ 1, a.err))) break;
            mbar_arrive_expect_tx(k_full0 + 8 * rk.s, kAttnPageBytes);
            tma_load_2d(k0 + rk.s * kAttnPageBytes, &tmKV, 0, row + h * 64, k_full0 + 8 * rk.s, pol);
            rk.next(kAttnKStages);
          }
          if (i > 0) {
            if (!(good = mbar_wait(v_empty0 + 8 * rv.s, rv.ph ^ 1, a.err))) break;
            mbar_arrive_expect_tx(v_full0 + 8 * rv.s, kAttnPageBytes);   // the ones rows stay
            tma_load_2d(v0 + rv.s * kAttnVStageBytes, &tmKV, 0, vrow + (a.Hkv + h) * 64, v_full0 + 8 * rv.s,
                        pol);
            rv.next(kAttnVStages);
          }
          vrow = row;
        }
        if (!good) {   // a wait ran out: the copies in flight land before the CTA ends
#pragma unroll 1
          for (int q = 0; q < kAttnKStages; ++q)
            mbar_wait(k_full0 + 8 * q, q < rk.s ? rk.ph : rk.ph ^ 1, a.err);
#pragma unroll 1
          for (int q = 0; q < kAttnVStages; ++q)
            mbar_wait(v_full0 + 8 * q, q < rv.s ? rv.ph : rv.ph ^ 1, a.err);
        }
      }
      first = __any_sync(0xFFFFFFFFu, first) != 0 && __all_sync(0xFFFFFFFFu, first) != 0;
      return __all_sync(0xFFFFFFFFu, good) != 0;
    };

    if (!a.early) pdl_wait();
    int np = 0, p_begin = 0, h = 0, safe = 0;   // the item being streamed (none yet)
    const int32_t* pt = nullptr;
#pragma unroll 1
    for (bool end = false; ok; ) {
      // stops: after page 5, three pages before the end, at the end (V^T of the
      // last page)
#pragma unroll 1
      for (int stop = 0, i0 = 0; ok && stop < 3; ++stop) {
        const int i1 = np == 0 ? 0 : (stop == 2 ? np + 1 : min(stop == 0 ? 5 : max(np - 2, 0), np + 1));
        if (i1 > i0) ok = stream(i0, i1, np, p_begin, safe, h, pt);
        i0 = max(i0, i1);
        if (ok && stop == 0 && tickets < published - 1) ok = ticket();
        if (ok && stop == 1 && np > 0) ask();
        if (ok && stop == 2) ok = fetch();
      }
      if (end || !ok) break;   // (the pass after the end took the last item's ticket)
      issued += np;
      ok = publish();
      np = nw.np;
      p_begin = nw.p_begin;
      h = nw.h;
      safe = nsafe;
      pt = npt;
      end = np == 0;
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
      RingPos ws, rk, rv, sb, pb;   // work slot; stages of the next S and PV; S and P buffers
      uint32_t item_ph = 0;         // q_full, o_free: one phase per item
      bool ok = true;
      auto issue_s = [&]() -> bool {
        if (!mbar_wait(k_full0 + 8 * rk.s, rk.ph, a.err)) return false;
        if (!mbar_wait(s_free0 + 8 * sb.s, sb.ph ^ 1, a.err)) return false;
        tc_fence_after();
        const uint64_t kdesc = kdesc0 + rk.s * (kAttnPageBytes >> 4);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          umma_f16(tmem + sb.s * 64, qdesc + 2 * k, kdesc + 2 * k, idesc, k > 0 ? 1u : 0u);
        umma_commit(s_full0 + 8 * sb.s);
        umma_commit(k_empty0 + 8 * rk.s);
        rk.next(kAttnKStages);
        sb.next(2);
        return true;
      };
#pragma unroll 1
      while (ok) {
        if (!mbar_wait(smem_u32(work_full) + 8 * ws.s, ws.ph, a.err)) break;
        const int np = work[ws.s].np;
        mbar_arrive(smem_u32(work_free) + 8 * ws.s);
        ws.next(2);
        if (np == 0) break;
        if (!mbar_wait(smem_u32(q_full), item_ph, a.err)) break;   // Q tile written
#pragma unroll 1
        for (int j = -1; j < np && ok; ++j) {
          if (j + 1 < np && !(ok = issue_s())) break;
          if (j < 0) continue;
          if (!(ok = mbar_wait(v_full0 + 8 * rv.s, rv.ph, a.err))) break;
          if (!(ok = mbar_wait(p_full0 + 8 * pb.s, pb.ph, a.err))) break;
          // the previous item's O has been read before this item's first P V
          if (j == 0 && !(ok = mbar_wait(smem_u32(o_free), item_ph ^ 1, a.err))) break;
          tc_fence_after();
          const uint64_t pdesc = pdesc0 + pb.s * (kAttnMaxRows * 128 >> 4);
          const uint64_t vdesc = vdesc0 + rv.s * (kAttnVStageBytes >> 4);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            umma_f16(tmem + 128, pdesc + 2 * k, vdesc + 2 * k, idesc_pv, (j > 0 || k > 0) ? 1u : 0u);
          umma_commit(v_empty0 + 8 * rv.s);
          rv.next(kAttnVStages);
          pb.next(2);
        }
        umma_commit(smem_u32(o_full));   // (also behind a failure: retires once every MMA above has)
        item_ph ^= 1;
      }
    }
  } else {
    // ---- softmax warps.  An item's descriptor stays in its slot until its rows
    // are out (registers are short: 168 a thread with two CTAs of six warps).
    AttnSync y{s_full, s_free, p_full, v_empty, sP, m_row};
    AttnRings rg;
    RingPos ws;
    uint32_t item_ph = 0, tick_ph = 0;
    bool owed = false;   // a ticket's answer is outstanding, for the item described by `pv`
    struct { const float* part; int nitems, R, tok0, h; } pv = {nullptr, 0, 0, 0, 0};
    int lim[4];
    auto wait_work = [&](RingPos q) {
      return __all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(work_full) + 8 * q.s, q.ph, a.err)) != 0;
    };
    pdl_wait();
    pdl_trigger();
    bool ok = true, have = false;   // have: the item in slot ws.s went through the softmax
    RingPos nx = ws;
#pragma unroll 1
    while (true) {
      // The next item.  Every S of the current one is done, so its Q tile is
      // free: the next Q goes there while the last P V completes, and its first
      // S follows.
      if (!(ok = wait_work(nx))) break;
      const int next_np = work[nx.s].np;
      if (next_np > 0) {
        const AttnWork& t = work[nx.s];
        const int R = t.R, tok0 = t.tok0;
        uint4 qv[8];
        attn_load_q(a, t.h, tok0, R, qv);
        attn_row_limits(a, warp, R, tok0, lim);
        attn_store_q(sQ, R, qv);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(q_full));
      }
      bool post = false;
      const AttnWork& w = work[ws.s];
      float* part = nullptr;
      if (have) {
        if (!(ok = __all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(o_full), item_ph, a.err)) != 0)) break;
        tc_fence_after();
        const uint32_t orow = tmem + (static_cast<uint32_t>(warp * 32) << 16) + 128;
        uint32_t o0[32], o1[32];
        tmem_ld32_nowait(orow, o0);
        tmem_ld32_nowait(orow + 32, o1);
        const uint32_t l1 = tmem_ld1(orow + 64);   // O's column 64: the row sums
        tmem_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(o_free));
        const int r = attn_block_row(threadIdx.x);   // block row
        auto O = [&](int k) { return __uint_as_float(k < 32 ? o0[k & 31] : o1[k & 31]); };
        const float l = __uint_as_float(l1);
        post = w.nitems > 1;
        part = a.part + (static_cast<size_t>(w.b) * a.Hkv + w.h) * a.max_items * kAttnMaxRows * kAttnRow;
        if (r < w.R) {
          if (post) {
            float* tile = part + static_cast<size_t>(w.c) * kAttnMaxRows * kAttnRow;
            float* dst = tile + r * 64;
#pragma unroll
            for (int k = 0; k < 64; k += 4)
              *reinterpret_cast<float4*>(dst + k) = make_float4(O(k), O(k + 1), O(k + 2), O(k + 3));
            *reinterpret_cast<float2*>(tile + kAttnTileMl + 2 * r) = make_float2(m_row[threadIdx.x], l);
          } else {   // the block's only item: its rows are final
            const float inv = 1.0f / l;
            const int tt = r * a.g_magic >> 16;
            const int hq = w.h * a.G + r - tt * a.G;
            __half* dst = a.out + (static_cast<size_t>(w.tok0 + tt) * a.Hq + hq) * 64;
#pragma unroll
            for (int cch = 0; cch < 8; ++cch) {
              uint32_t w4[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                __half2 hv = __floats2half2_rn(O(8 * cch + 2 * e) * inv, O(8 * cch + 2 * e + 1) * inv);
                w4[e] = *reinterpret_cast<uint32_t*>(&hv);
              }
              *reinterpret_cast<uint4*>(dst + 8 * cch) = make_uint4(w4[0], w4[1], w4[2], w4[3]);
            }
          }
        }
        item_ph ^= 1;
      }
      // the previous item's ticket, then this item's rows to theirs; behind the
      // last item its own ticket too
#pragma unroll 1
      while (true) {
        if (owed) {
          owed = false;
          if (!(ok = __all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(tick_full), tick_ph, a.err)) != 0)) break;
          tick_ph ^= 1;
          if (*tick) {   // the last item: merge (every P V so far has retired: the P tiles are free)
            ok = attn_merge_rows(pv.part, reinterpret_cast<float*>(sP), a.out, merge_bar, pv.nitems, pv.R,
                                 pv.tok0, pv.h, a.Hq, a.G, a.g_magic, a.err);
            if (!ok) break;
          }
        }
        __syncwarp();
        if (post) {
          if (lane == 0) mbar_arrive(smem_u32(rows_full));
          pv = {part, w.nitems, w.R, w.tok0, w.h};
          owed = true;
          post = false;
          if (next_np == 0) continue;
        }
        break;
      }
      if (!ok) break;
      if (have) {
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(work_free) + 8 * ws.s);
      }
      if (next_np == 0) break;
      ws = nx;
      nx.next(2);
      have = true;
      {
        const int R = work[ws.s].R, rows_w = warp < R ? (R - warp + 3) / 4 : 0;   // rows in this warp's quarter
        ok = attn_softmax(a, y, tmem, warp, (rows_w + 7) / 8, next_np, work[ws.s].p_begin, lim, rg);
      }
      __syncwarp();   // m_row is written and read by one warp
      if (!ok) break;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kAttnMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, kAttnTmemCols);
  }
}

}  // namespace gs
