// gemm_wide.cuh -- persistent tcgen05 GEMM for everything that does not split K
// across CTAs: wide decode windows (K reduced in fixed chunks), prefill chunks
// and the LM head.
//
// One CTA per SM walks tiles of 128 weight rows x BN token rows (token tiles
// fastest, so neighbouring CTAs share a weight tile).  The grid has a CTA per
// tile; a running CTA takes over CTAs that have not started (cluster launch
// control), so SMs that get less bandwidth take fewer tiles: with a fixed share
// per SM the LM head at 17 rows took 20 or 40 us, by where its weights lay.
//   warps 0, 2  TMA producers of the weight and the token rows: k-blocks of all
//             tiles, one after the other, through one ring of shared-memory
//             stages (they run ahead across tiles)
//   warp 1    MMA issuer: chunk after chunk into a ring of TMEM buffers; a
//             buffer is reused once the epilogue warps have drained it
//             (a single token tile that fits, as the LM head's at decode, is
//             loaded once and stays: 464 tiles re-reading the same 34 KB had
//             152 SMs waiting on the few L2 slices that hold it, 28 or 47 us by
//             where the buffers lay)
//   warp 3    scheduler: asks for the next tile and hands it to the other roles
//   others    one or two groups of four epilogue warps, each owning BN / NG of
//             a tile's token columns
// K is reduced as `chunks` chunks, each summed from zero in k order, then the
// chunks added in order from zero -- the same sums, in the same order, as
// split-K across the CTAs of a cluster, so a row's bits do not depend on the
// window.  A group keeps its running sum in registers (CW = BN / NG columns a
// thread), writes the total over the last chunk's TMEM buffer and runs the
// shared epilogue on 32-token slices of it, while the MMAs of the next tile
// fill the other buffers.
//
// What bounds it: the ring.  Per 64-deep k-block, all 152 SMs running (K 8192 less K
// 2048): 253 cycles at BN 32, 80 bytes per clock and SM from L2; 310 at 64 under
// SwiGLU, 397 under the epilogues whose fp32 slices leave a stage less; 417 at 96; 435
// / 460 at 144; 545 / 630 at 192; 720 / 840 at 256, where the MMA rate is 515.  One
// CTA per tile instead paid its start-up, its first load latency and its
// epilogue per tile: 544 rows of gate/up took 24.5 us, LM head at 17 rows 30 us,
// a 4096-row prefill gate/up 100 us; here 19.0, 26.6 (23.6 as a graph node, 76% of
// the measured copy rate) and 57-59 us.  (The 256-row residual kernel spills 32
// bytes beyond its 168 registers; the others none.)
#pragma once
#include "gemm_tc.cuh"

namespace gs {

template <int BN>
struct WideShape {
  static constexpr int kKB = BN <= 96 ? 2 : 1;          // k-blocks per stage (at most)
  static constexpr int kABlock = 128 * 128;             // one 64-deep k-block of W
  static constexpr int kBBlock = BN * 128;              // and of X
  static constexpr int kStageBytes = kKB * (kABlock + kBBlock);
  static constexpr int kGroups = BN >= 64 ? 2 : 1;      // epilogue groups of four warps
  static constexpr int kCols = BN / kGroups;            // token columns of a group
  static constexpr int kThreads = 128 + kGroups * 128;
  static constexpr int kBufCols = (BN + 31) / 32 * 32;  // TMEM columns of a chunk buffer
  static constexpr int kBufs = 512 / kBufCols < 4 ? 512 / kBufCols : 4;
  static constexpr int kTmemCols = kBufs * kBufCols <= 128 ? 128 : (kBufs * kBufCols <= 256 ? 256 : 512);
  // a group's epilogue slice: fp16 [32][72] for SwiGLU, else fp32 [32][132] and
  // the residual's partial sums [32][16]
  __host__ __device__ static constexpr int xs_bytes(int epi) {
    return epi == kEpiSwiGLU ? 32 * 72 * 2 : (32 * 132 + 32 * 16) * 4;
  }
  static constexpr bool kStageRope = BN <= 64;
  static constexpr int kBarBytes = 512;
  static constexpr int kSched = 2;                      // scheduler answers kept
  __host__ __device__ static constexpr int tail_bytes(int epi) {
    return kGroups * xs_bytes(epi) + kBarBytes + 16 * BN + (kStageRope && epi == kEpiQKV ? BN * 256 : 0);
  }
  __host__ __device__ static constexpr int stages(int epi) {
    const int s = (227 * 1024 - 1024 - tail_bytes(epi)) / kStageBytes;
    return s < 10 ? s : 10;
  }
  __host__ __device__ static constexpr int ring_bytes(int epi) { return stages(epi) * kStageBytes; }
  __host__ __device__ static constexpr int smem_bytes(int epi) {
    return 1024 + ring_bytes(epi) + tail_bytes(epi);
  }
  // With one token tile, the token rows of all nkb k-blocks may stay in shared
  // memory and the ring hold weights only: the stages that leaves (0: too few).
  __host__ __device__ static constexpr int resident_stages(int epi, int nkb) {
    const int left = ring_bytes(epi) - nkb * kBBlock;
    const int st = left > 0 ? left / (kKB * kABlock) : 0;
    return st < 3 ? 0 : (st < 10 ? st : 10);
  }
  static_assert(kStageBytes % 1024 == 0, "stages keep the swizzle atom's alignment");
  static_assert(xs_bytes(kEpiArgmax) >= 32 * 129 * 4 + 4 * 32 * 8 + 2 * 4 * 32 * 4, "argmax slice");
  static_assert((2 * 10 + 2 * 4 + 2 * kSched + 1) * 8 + 16 + 16 * kSched <= kBarBytes, "barriers");
  static_assert(kCols % 8 == 0 && kBufs >= 2 && stages(kEpiQKV) >= 2, "tile shape");
};

// N fp32 columns of this thread's TMEM lane, N a multiple of 8 (no wait).
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                 "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
               "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

// OR of a predicate over the 128 threads of an epilogue group.
__device__ __forceinline__ bool group_any(bool v, int bar) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "barrier.red.or.pred p, %2, 128, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"(v ? 1u : 0u), "r"(bar)
      : "memory");
  return r != 0;
}

// XRES: the launch's single token tile stays in shared memory.
template <int BN, int EPI, bool XRES>
__global__ void __launch_bounds__(WideShape<BN>::kThreads, 1)
    gemm_wide_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                     const GemmArgs a) {
  using S = WideShape<BN>;
  constexpr int NB = S::kBufs, CW = S::kCols, KB = S::kKB;
  // stage: W blocks, then X blocks; or W blocks only, and X after the ring
  const int NS = XRES ? S::resident_stages(EPI, a.K / 64) : S::stages(EPI);
  constexpr uint32_t stage_stride = XRES ? KB * S::kABlock : S::kStageBytes;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* tail = smem + S::ring_bytes(EPI);
  float* xs_all = reinterpret_cast<float*>(tail);
  uint64_t* bars = reinterpret_cast<uint64_t*>(tail + S::kGroups * S::xs_bytes(EPI));
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * NS;
  const uint32_t acc_full0 = empty0 + 8 * NS, acc_free0 = acc_full0 + 8 * NB;
  const uint32_t clc_full0 = acc_free0 + 8 * NB, clc_free0 = clc_full0 + 8 * S::kSched;
  const uint32_t go0 = clc_free0 + 8 * S::kSched;   // the weight producer nears its tile's end
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * NS + 2 * NB + 2 * S::kSched + 1);
  const uint32_t clc_slot0 = smem_u32(bars) + S::kBarBytes - 16 * S::kSched;   // 16-byte aligned
  float* rs_all = reinterpret_cast<float*>(tail + S::kGroups * S::xs_bytes(EPI) + S::kBarBytes);   // [BN]
  int* pos_all = reinterpret_cast<int*>(rs_all + BN);                                         // [BN]
  long long* kvdst_all = reinterpret_cast<long long*>(pos_all + BN);                          // [BN]
  float2* cs_all = reinterpret_cast<float2*>(kvdst_all + BN);                                 // [BN][32]
  const uint32_t stage0 = smem_u32(smem);

  const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0);   // warp-uniform
  const int lane = threadIdx.x & 31;
  const int nchunk = a.chunks > 1 ? a.chunks : 1;
  const int kpc = a.K / 64 / nchunk;               // k-blocks per chunk
  const int kps = (KB == 2 && kpc % 2 == 0) ? 2 : 1;   // k-blocks per stage
  const int steps = kpc / kps;                     // stages per chunk

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmW);
    tma_prefetch_desc(&tmX);
#pragma unroll 1
    for (int s = 0; s < 2 * NS + NB; ++s) mbar_init(full0 + 8 * s, s < NS ? 2 : 1);   // full: W and X
#pragma unroll 1
    for (int b = 0; b < NB; ++b) mbar_init(acc_free0 + 8 * b, 4 * S::kGroups);
    mbar_init(go0, 1);
    for (int b = 0; b < S::kSched; ++b) {
      mbar_init(clc_full0 + 8 * b, 1);
      mbar_init(clc_free0 + 8 * b, 3 + 4 * S::kGroups);   // two producers, MMA, epilogue warps
    }
    fence_mbar_init();
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), S::kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // The next tile: 1 and *tile, 0 if there is none, -1 if the wait ran out.
  // Called by one thread or a whole warp; `arrive` posts that the slot was read.
  auto next_tile = [&](RingPos& q, int* tile, bool arrive) -> int {
    if (!mbar_wait(clc_full0 + 8 * q.s, q.ph, a.err)) return -1;
    int y, z;
    const bool more = clc_answer(clc_slot0 + 16 * q.s, tile, &y, &z);
    fence_proxy_async_smem();   // read before the slot's next answer is written
    if (arrive) mbar_arrive(clc_free0 + 8 * q.s);
    q.next(S::kSched);
    return more ? 1 : 0;
  };

  if (warp == 3) {
    pdl_wait();
    pdl_trigger();
    if (elect_one()) {
      // A tile is asked for when the weight producer has a ring's worth of its
      // tile left: early enough for the answer, late enough that a slow SM does
      // not hold tiles it has not begun.
      RingPos q;
      uint32_t go_ph = 0;
      int tile;
#pragma unroll 1
      for (; ; go_ph ^= 1) {
        if (!mbar_wait(go0, go_ph, a.err)) break;
        if (!mbar_wait(clc_free0 + 8 * q.s, q.ph ^ 1, a.err)) break;
        mbar_arrive_expect_tx(clc_full0 + 8 * q.s, 16);
        clc_try_cancel(clc_slot0 + 16 * q.s, clc_full0 + 8 * q.s);
        if (next_tile(q, &tile, false) != 1) break;
      }
    }
  } else if (warp == 0 || warp == 2) {
    const bool is_w = warp == 0;
    if (is_w ? elect_one() : (pdl_wait(), pdl_trigger(), elect_one())) {
      // ---- TMA producers: one thread for the weight rows (its first stages go
      // out before the dependency wait, which it never needs), one for the token
      // rows.
      const uint64_t pol = is_w ? l2_policy_evict_first() : l2_policy_evict_last();
      const uint32_t bytes = static_cast<uint32_t>(kps) * (is_w ? S::kABlock : S::kBBlock);
      const uint32_t block = is_w ? S::kABlock : S::kBBlock;
      const uint32_t x0 = stage0 + (XRES ? NS * stage_stride : KB * S::kABlock);
      const int per_tile = nchunk * steps;
      const int ask = per_tile > NS ? per_tile - NS : 0;
      RingPos r;
      r.ph = 1;   // a fresh stage counts as released
      RingPos q;
      bool ok = true;
      int tile = blockIdx.x;
      bool first = true;
#pragma unroll 1
      for (int more = 1; more == 1 && ok; first = false) {
        const int feat = tile / a.tok_tiles;
        const int xrow = a.x_row0 + (tile - feat * a.tok_tiles) * BN;
#pragma unroll 1
        for (int i = 0; i < per_tile; ++i, r.next(NS)) {
          if (!mbar_wait(empty0 + 8 * r.s, r.ph, a.err)) {
            ok = false;
            break;
          }
          if (is_w && i == ask) mbar_arrive(go0);
          const uint32_t fb = full0 + 8 * r.s;
          if (!is_w && XRES && !first) {   // these rows are there already
            mbar_arrive(fb);
            continue;
          }
          uint32_t dst = is_w ? stage0 + r.s * stage_stride
                              : x0 + (XRES ? i * kps * S::kBBlock : r.s * stage_stride);
          mbar_arrive_expect_tx(fb, bytes);
#pragma unroll 1
          for (int k = 0; k < kps; ++k, dst += block) {
            const int kx = (i * kps + k) * 64;
            if (!is_w) tma_load_2d(dst, &tmX, kx, xrow, fb, pol);
            else if constexpr (EPI == kEpiSwiGLU) tma_load_4d(dst, &tmW, kx, 0, 0, feat * 4, fb, pol);
            else tma_load_2d(dst, &tmW, kx, feat * 128, fb, pol);
          }
        }
        if (ok) more = next_tile(q, &tile, true);
      }
      if (!ok) {   // a wait ran out: the copies in flight land before the CTA ends
#pragma unroll 1
        for (int s = 0; s < NS; ++s)
          mbar_wait(full0 + 8 * s, s < r.s ? r.ph ^ 1 : r.ph, a.err);
      }
    }
    if (is_w) {
      __syncwarp();
      pdl_wait();
      pdl_trigger();
    }
  } else if (warp == 1) {
    pdl_wait();
    pdl_trigger();
    if (elect_one()) {
      // ---- MMA issuer, N = the tile's rows rounded up to 16 (a ragged last
      // tile issues narrower MMAs; its columns past M are never used)
      const uint64_t ad0 = umma_desc_sw128(stage0);
      const uint64_t bd0 = umma_desc_sw128(stage0 + (XRES ? NS * stage_stride : KB * S::kABlock));
      RingPos r, b, t;
      bool ok = true;
      int used = 0;   // chunks issued
      int tile = blockIdx.x;
#pragma unroll 1
      for (int more = 1; more == 1 && ok; ) {
        const int rows = min(BN, a.M - (tile % a.tok_tiles) * BN);
        const uint32_t idesc = umma_idesc_f16(128, (rows + 15) / 16 * 16);
#pragma unroll 1
        for (int c = 0; c < nchunk && ok; ++c, ++used) {
          if (used >= NB && !mbar_wait(acc_free0 + 8 * b.s, b.ph ^ 1, a.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t dst = tmem + b.s * S::kBufCols;
#pragma unroll 1
          for (int i = 0; i < steps; ++i, r.next(NS)) {
            if (!mbar_wait(full0 + 8 * r.s, r.ph, a.err)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t ad = ad0 + r.s * (stage_stride >> 4);
            const uint64_t bd = bd0 + (XRES ? (c * steps + i) * kps * (S::kBBlock >> 4)
                                             : r.s * (stage_stride >> 4));
#pragma unroll
            for (int q = 0; q < 4; ++q)
              umma_f16(dst, ad + 2 * q, bd + 2 * q, idesc, (i > 0 || q > 0) ? 1u : 0u);
            if (kps == 2) {
#pragma unroll
              for (int q = 0; q < 4; ++q)
                umma_f16(dst, ad + (S::kABlock >> 4) + 2 * q, bd + (S::kBBlock >> 4) + 2 * q, idesc, 1u);
            }
            umma_commit(empty0 + 8 * r.s);
          }
          if (ok) umma_commit(acc_full0 + 8 * b.s);
          b.next(NB);
        }
        if (ok) more = next_tile(t, &tile, true);
      }
    }
  } else {
    // ---- epilogue group g: token columns [g CW, (g + 1) CW) of every tile
    const int g = S::kGroups == 2 ? (warp - 4) >> 2 : 0;
    const int quarter = warp & 3;               // TMEM lanes this warp can read
    const int row = quarter * 32 + lane;        // weight row of the tile
    const int bar_a = 1 + 2 * g, bar_b = 2 + 2 * g;
    float* xs = xs_all + g * (S::xs_bytes(EPI) / 4);
    float* rs_s = rs_all + g * CW;
    int* pos_s = pos_all + g * CW;
    long long* kvdst_s = kvdst_all + g * CW;
    float2* cs_s = S::kStageRope ? cs_all + g * CW * 32 : nullptr;
    const uint32_t trow = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + g * CW;
    bool waited = false;   // griddepcontrol.wait done
    bool ok = true;
    RingPos b, t;
    int tile = blockIdx.x;
#pragma unroll 1
    while (true) {
      const int feat = tile / a.tok_tiles;
      const int tok0 = (tile - feat * a.tok_tiles) * BN + g * CW;   // the group's first token
      const int ntok = min(CW, a.M - tok0);                         // may be <= 0: nothing to produce
      // per-token data, while the tile's MMAs run.  Positions, page-table rows
      // and the RoPE table are written by kernels that completed before the
      // previous one started: the first tile's are read before the wait.
      if constexpr (EPI == kEpiQKV) {
        for (int t = row; t < ntok; t += 128) {
          long long dst = -1;
          const int p = a.pos[tok0 + t];
          const int slot = a.tok_slot[tok0 + t];
          if (slot >= 0) {
            const int lp = p >> 6;
            const int phys = (p >= 0 && p < a.max_ctx && lp < a.pt_stride)
                                 ? a.page_table[static_cast<size_t>(slot) * a.pt_stride + lp] : -1;
            if (phys < 0 || phys >= a.n_pages) atomicExch(a.err, kErrBounds);
            else dst = static_cast<long long>(phys) * 2 * a.Hkv * 4096 + (p & 63) * 64;
          }
          kvdst_s[t] = dst;
          pos_s[t] = p;
          if constexpr (S::kStageRope) {
            if (p >= 0 && p < a.max_ctx) {
              const float4* src = reinterpret_cast<const float4*>(a.rope + static_cast<size_t>(p) * 32);
              float4* dstv = reinterpret_cast<float4*>(cs_s + t * 32);
#pragma unroll 4
              for (int q = 0; q < 16; ++q) dstv[q] = src[q];
            }
          }
        }
      }
      if (!waited) {
        pdl_wait();
        pdl_trigger();
        waited = true;
      }
      if (a.ssp_in != nullptr) {
        // folded-norm scale from the previous kernel's per-tile sums of h^2
        for (int t = row; t < ntok; t += 128) {
          const float* sp = a.ssp_in + static_cast<size_t>(a.x_row0 + tok0 + t) * a.n_ssp;
          float part[16], ss = 0.f;
#pragma unroll
          for (int q = 0; q < 16; ++q) part[q] = q < a.n_ssp ? sp[q] : 0.f;
#pragma unroll
          for (int q = 0; q < 16; ++q) ss += part[q];
          for (int q = 16; q < a.n_ssp; ++q) ss += sp[q];
          rs_s[t] = rsqrtf(ss * a.inv_d + a.eps) * a.w_scale;
        }
      }
      // the chunks: running sum in registers, its total over the last buffer
      if (nchunk > 1) {
        uint32_t sum[CW];
#pragma unroll
        for (int j = 0; j < CW; ++j) sum[j] = 0u;
#pragma unroll 1
        for (int c = 0; c < nchunk; ++c) {
          if (ok) ok = __all_sync(0xFFFFFFFFu, mbar_wait(acc_full0 + 8 * b.s, b.ph, a.err)) != 0;
          tc_fence_after();
          const uint32_t buf = trow + b.s * S::kBufCols;
#pragma unroll
          for (int j0 = 0; j0 < CW; j0 += 24) {
            constexpr int kStep = 24;
            uint32_t ch[kStep];
#pragma unroll
            for (int j = 0; j < kStep; j += 8)
              if (j0 + j < CW) tmem_ld8_nowait(buf + j0 + j, ch + j);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < kStep; ++j)
              if (j0 + j < CW)
                sum[j0 + j] = __float_as_uint(__uint_as_float(sum[j0 + j]) + __uint_as_float(ch[j]));
          }
          if (c + 1 < nchunk) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_free0 + 8 * b.s);
            b.next(NB);
          } else {
#pragma unroll
            for (int j = 0; j < CW; j += 8) tmem_st8(buf + j, sum + j);
            tmem_wait_st();
          }
        }
      } else {
        if (ok) ok = __all_sync(0xFFFFFFFFu, mbar_wait(acc_full0 + 8 * b.s, b.ph, a.err)) != 0;
        tc_fence_after();
      }
      // one barrier: the per-token data is visible, and a wait that ran out in
      // any warp of the group ends the group together
      if (group_any(!ok, bar_a)) break;
      const uint32_t buf = trow + b.s * S::kBufCols;
#pragma unroll 1
      for (int c = 0; c < ntok; c += 32) {
        float v[32];
        if constexpr (CW % 32 == 0) {
          tmem_ld_32x32b_x32(buf + c, v);
        } else {   // a last slice of 8 columns reads its own columns only
          uint32_t u[32];
#pragma unroll
          for (int j = 0; j < 32; j += 8)
            tmem_ld8_nowait(buf + min(c + j, CW - 8), u + j);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(u[j]);
        }
        const TokMeta tm{a.ssp_in ? rs_s + c : nullptr, kvdst_s + c, pos_s + c,
                         cs_s ? cs_s + c * 32 : nullptr};
        gemm_epilogue<EPI>(a, v, ntok - c <= 8 ? 8 : 32, row, feat, tok0 + c, 0, min(32, ntok - c), xs,
                           tm, bar_a, bar_b);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_free0 + 8 * b.s);
      b.next(NB);
      // the group leaves together, also when a wait ran out in one of its warps
      int more = next_tile(t, &tile, false);
      __syncwarp();
      if (lane == 0) mbar_arrive(clc_free0 + 8 * (t.s == 0 ? S::kSched - 1 : t.s - 1));
      if (group_any(more < 0, bar_b) || more != 1) break;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, S::kTmemCols);
}

}  // namespace gs
