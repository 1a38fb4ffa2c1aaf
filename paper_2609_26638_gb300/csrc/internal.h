// internal.h -- declarations shared by the library's translation units.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

namespace gs {

struct GemmArgs;

// cudaLaunchKernelEx with optional programmatic stream serialisation (PDL) and
// an optional thread-block cluster shape.
template <typename... KArgs, typename... Args>
cudaError_t launch_ex(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                      cudaStream_t s, bool pdl, dim3 cluster, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attrs[2];
  int n = 0;
  if (pdl) {
    attrs[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  if (cluster.x * cluster.y * cluster.z > 1) {
    attrs[n].id = cudaLaunchAttributeClusterDimension;
    attrs[n].val.clusterDim.x = cluster.x;
    attrs[n].val.clusterDim.y = cluster.y;
    attrs[n].val.clusterDim.z = cluster.z;
    ++n;
  }
  cfg.attrs = attrs;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// SMs of one GB300 (two dies x 76).  Work decompositions that must not depend
// on the device (the split-K factors) use this constant, not a query.
constexpr int kNumSMs = 152;
// GemmEpilogue's values, for the dispatch rules.
constexpr int kEpiSwiGLUKind = 2, kEpiQKVKind = 4;

// Token tile of a GEMM over T token rows that splits K across CTAs.
inline int gemm_bn_for(int T) { return T <= 32 ? 32 : (T <= 64 ? 64 : (T <= 128 ? 128 : 256)); }

// Launch Y = epilogue(W . X^T) for one weight matrix.  grid = (feat_tiles,
// tok_tiles, splits).  Returns a cudaError_t.
// Split-K partials are reduced through distributed shared memory inside a
// cluster of the `splits` CTAs of a tile when splits <= kMaxClusterSplits,
// else through global scratch by the last CTA to arrive (same order, same bits).
constexpr int kMaxClusterSplits = 8;
// The cluster reduction gives split CTA q the tokens [q*per, (q+1)*per) of a
// BN-token tile, per = BN / splits, and its epilogue handles per <= 8 or a
// per that divides 32 (a slice never straddles a 32-token chunk).
inline bool gemm_cluster_ok(int bn, int splits) {
  if (splits < 2 || splits > kMaxClusterSplits || bn > 64 || bn % splits) return false;
  const int per = bn / splits;
  return per <= 8 || 32 % per == 0;
}
// Token tiles of the persistent GEMM (splits == 1).
constexpr int kWideTiles = 6;
constexpr int kWideBN[kWideTiles] = {32, 64, 96, 144, 192, 256};

// The decoder's token maps: one per tile of either kernel.
constexpr int kTokenMaps = kWideTiles + 1;
constexpr int kTokenMapBN[kTokenMaps] = {32, 64, 96, 144, 192, 256, 128};

inline int token_map_index(int bn) {
  for (int i = 0; i < kTokenMaps; ++i)
    if (kTokenMapBN[i] == bn) return i;
  return -1;
}

// The token tile with the least estimated time: rounds of tiles over the SMs, each a
// start, its k-blocks and its epilogue, which share the SM (the longer and 0.63 of the
// shorter).  The wider on a tie.  Cycles, fitted to 950 launches of every tile (four
// epilogues, 68-4,096 rows, 256-59,392 features, K 64-8,192, 1-8 chunks): the choice
// is 0.2% from the fastest tile in the mean and 8% at worst; one k-block and one
// slice cost for all epilogues, made from long SwiGLU launches, was 3% and 121%
// (fp16 stores of 4,096 x 16,384, K 448: 154 us with 64-row tiles, 70 with 256).
// SwiGLU's fp16 slices leave the ring a stage more than the others' fp32 ones; a
// chunk of an odd number of k-blocks fills half of a stage of two (32-96 rows); the
// epilogue warps add up each chunk.
inline int wide_bn(int epi, int feat_tiles, int T, int nkb, int chunks) {
  constexpr double kBlock[2][kWideTiles] = {{207, 315, 388, 387, 586, 779}, {317, 394, 585, 611, 778, 1025}};
  constexpr double kEpilogue[5][kWideTiles] = {{229, 1581, 1946, 3891, 5282, 8176},       // fp16 stores
                                               {705, 2131, 6204, 10984, 14755, 25536},    // residual
                                               {1185, 1350, 7219, 10301, 10664, 13872},   // SwiGLU
                                               {1644, 1858, 6787, 10436, 11981, 17982},   // argmax
                                               {229, 1581, 1946, 3891, 5282, 8176}};      // QKV, as stores
  const int n = chunks > 1 ? chunks : 1;
  const bool odd = nkb / n % 2 != 0;
  int best = 32;
  double best_cost = -1;
  for (int i = kWideTiles - 1; i >= 0; --i) {
    const int bn = kWideBN[i];
    const long long tiles = static_cast<long long>(feat_tiles) * ((T + bn - 1) / bn);
    const long long rounds = (tiles + kNumSMs - 1) / kNumSMs;
    const double main = nkb * kBlock[epi == kEpiSwiGLUKind][i] * (odd && bn <= 96 ? 1.38 : 1.0);
    const double epilogue = kEpilogue[epi][i] + 0.7 * (n - 1) * bn;
    const double cost = rounds * (main > epilogue ? main + 0.63 * epilogue + 3478 : epilogue + 0.63 * main + 3478);
    if (best_cost < 0 || cost < best_cost) {
      best_cost = cost;
      best = bn;
    }
  }
  return best;
}

// Unsplit launches of a little more than one wave of long tiles, one token tile:
// the persistent kernel's one CTA per SM takes a second round of tiles on a few SMs,
// where a CTA per tile, two on an SM, all start together (gemm_tc_kernel).
// Measured, persistent / CTA per tile: 154 feature tiles x K 4096 34.7 / 29.8 us at
// 17 rows, 39.8 / 32.1 at 64, 42.6 / 35.3 at 128; 190 x 8192 66.7 / 64.0, 77.9 / 68.3,
// 81.5 / 72.6; 216 x 1024 14.4 / 13.3, 16.5 / 14.4, 18.9 / 17.0; even at 250, slower
// at 152 and from 304 on.  193-256 rows, whose 256-row tiles have the shorter ring
// beside the epilogue's slices, from K 8192 on and up to two tiles per SM: 154
// feature tiles 109 / 93, 290 120 / 114 (at K 4096 48.9 / 51.6).
inline bool cta_per_tile(int epi, int feat_tiles, int T, int nkb) {
  if (feat_tiles <= kNumSMs) return false;
  if (T <= (epi == kEpiQKVKind ? 64 : 128)) return 2 * feat_tiles <= 3 * kNumSMs;
  return epi != kEpiQKVKind && T > 192 && T <= 256 && nkb >= 128 && feat_tiles <= 2 * kNumSMs;
}
// Token tile of a launch that does not split K across CTAs.
inline int unsplit_bn(int epi, int feat_tiles, int T, int nkb, int chunks) {
  return chunks <= 1 && cta_per_tile(epi, feat_tiles, T, nkb) ? gemm_bn_for(T) : wide_bn(epi, feat_tiles, T, nkb, chunks);
}

cudaError_t launch_gemm(int bn, int epi, const CUtensorMap& tmW, const CUtensorMap& tmX,
                        const GemmArgs& args, int feat_tiles, int tok_tiles, cudaStream_t s,
                        bool pdl = false);

// Zero n words on the stream with a kernel that lets a dependent launch (PDL)
// start its prologue at once: a launch after it costs about 3 us less than after
// a memset node, whose completion the next kernel's launch waits for.
cudaError_t clear_words(int* p, size_t n, cudaStream_t s);

// The persistent kernel (args.splits == 1, bn one of kWideBN).
cudaError_t launch_gemm_wide(int bn, int epi, const CUtensorMap& tmW, const CUtensorMap& tmX,
                             const GemmArgs& args, int feat_tiles, int tok_tiles, cudaStream_t s,
                             bool pdl);

// 2-D fp16 tensor map over a row-major [rows, cols] array, box {64 columns,
// box_rows rows}, 128-byte swizzle, zero fill out of bounds.  The driver's
// encoder is looked up once per process (thread-safe).  False if the lookup
// or the encode fails.
bool make_map(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows);
// The map of a SwiGLU weight [2 N, K] (gate rows, then up rows): one box holds
// the 128 rows of 64 output features in four groups of 16 gate rows and their
// 16 up rows, so the two rows of a feature land in one warp's TMEM lanes.
// N % 64 == 0.
bool make_map_swiglu(CUtensorMap* m, const void* base, uint64_t N, uint64_t K);

// Sets the dynamic shared-memory limit of every GEMM instantiation once.
cudaError_t gemm_init_attributes();
cudaError_t gemm_wide_init_attributes();
// Every kernel's launch attributes on the current device, once per device
// (thread-safe); call before the first launch.
cudaError_t ensure_kernel_attributes();

}  // namespace gs
