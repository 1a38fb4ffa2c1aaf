// gemm.cu -- launcher of the GEMM and instantiations of its split-K kernel.
#include "gemm_tc.cuh"
#include "internal.h"

namespace gs {

static __global__ void clear_words_kernel(int* p, unsigned n) {
  pdl_trigger();
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = 0;
}

cudaError_t clear_words(int* p, size_t n, cudaStream_t s) {
  return launch_ex(clear_words_kernel, dim3(static_cast<unsigned>((n + 255) / 256)), dim3(256), 0, s, false,
                   dim3(1), p, static_cast<unsigned>(n));
}

template <int BN, int EPI>
static cudaError_t launch_one(const CUtensorMap& tmW, const CUtensorMap& tmX, GemmArgs a,
                              int feat_tiles, int tok_tiles, cudaStream_t s, bool pdl) {
  using S = GemmShape<BN>;
  // Pipeline depth, never more than the k-blocks one CTA loads.  Decode
  // windows (up to 64 rows): a fixed depth that leaves room for a second
  // resident CTA and for the neighbouring kernels' CTAs that overlap it under
  // programmatic dependent launch.  Wider launches stream K through each CTA: the
  // deepest pipeline that still fits the CTAs one SM holds (one when the grid
  // is at most one CTA per SM, else two), since bytes in flight per SM set
  // their load rate; the same for unsplit launches.  Clusters always two: with one CTA per SM a cluster of 8
  // waits for 8 empty SMs of one GPC (1024 x 4096 weight, 68 rows, 128 CTAs:
  // 17.4 us in the decoder's graph, 13.3 with two).
  const bool cl = a.splits > 1 && a.cluster;
  int want = S::kStagesDefault;
  if (a.M > 64 || a.splits == 1)
    want = S::stages_fitting(
        !cl && static_cast<long>(feat_tiles) * tok_tiles * a.splits <= kNumSMs ? 1 : 2, EPI, cl);
  const int kb = a.kb_per_split;
  a.stages = kb < S::kStagesMin ? S::kStagesMin : (kb > want ? want : kb);
  dim3 grid(tok_tiles, feat_tiles, a.splits);
  const size_t smem = S::smem_bytes(a.stages, EPI, cl);
  if constexpr (S::kClusterOk) {
    if (cl)
      return launch_ex(gemm_tc_kernel<BN, EPI, kTcCluster>, grid, dim3(128), smem, s, pdl, dim3(1, 1, a.splits),
                       tmW, tmX, a);
  }
  if (a.splits == 1)
    return launch_ex(gemm_tc_kernel<BN, EPI, kTcWhole>, grid, dim3(128), smem, s, pdl, dim3(1, 1, 1), tmW, tmX,
                     a);
  return launch_ex(gemm_tc_kernel<BN, EPI, kTcScratch>, grid, dim3(128), smem, s, pdl, dim3(1, 1, 1), tmW, tmX,
                   a);
}

template <int BN>
static cudaError_t launch_bn(int epi, const CUtensorMap& tmW, const CUtensorMap& tmX,
                             const GemmArgs& a, int ft, int tt, cudaStream_t s, bool pdl) {
  switch (epi) {
    case kEpiStoreF16: return launch_one<BN, kEpiStoreF16>(tmW, tmX, a, ft, tt, s, pdl);
    case kEpiResidF32: return launch_one<BN, kEpiResidF32>(tmW, tmX, a, ft, tt, s, pdl);
    case kEpiSwiGLU: return launch_one<BN, kEpiSwiGLU>(tmW, tmX, a, ft, tt, s, pdl);
    case kEpiArgmax: return launch_one<BN, kEpiArgmax>(tmW, tmX, a, ft, tt, s, pdl);
    case kEpiQKV:   // the decoder's own launches: tiles of 32 and 64
      if constexpr (BN <= 64) return launch_one<BN, kEpiQKV>(tmW, tmX, a, ft, tt, s, pdl);
      break;
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_gemm(int bn, int epi, const CUtensorMap& tmW, const CUtensorMap& tmX,
                        const GemmArgs& a, int feat_tiles, int tok_tiles, cudaStream_t s,
                        bool pdl) {
  static_assert(kEpiStoreF16 == 0 && kEpiResidF32 == 1 && kEpiSwiGLUKind == kEpiSwiGLU && kEpiArgmax == 3 &&
                    kEpiQKVKind == kEpiQKV, "the dispatch rules' names");
  if (a.splits == 1 && (a.chunks > 1 || !cta_per_tile(epi, feat_tiles, a.M, a.K / 64)))
    return launch_gemm_wide(bn, epi, tmW, tmX, a, feat_tiles, tok_tiles, s, pdl);
  switch (bn) {
    case 32: return launch_bn<32>(epi, tmW, tmX, a, feat_tiles, tok_tiles, s, pdl);
    case 64: return launch_bn<64>(epi, tmW, tmX, a, feat_tiles, tok_tiles, s, pdl);
    case 128: return launch_bn<128>(epi, tmW, tmX, a, feat_tiles, tok_tiles, s, pdl);
    case 256: return launch_bn<256>(epi, tmW, tmX, a, feat_tiles, tok_tiles, s, pdl);
  }
  return cudaErrorInvalidValue;
}

template <int BN, int EPI>
static cudaError_t set_attr_one() {
  constexpr int bytes = GemmShape<BN>::kSmemMax;
  cudaError_t e = cudaSuccess;
  if constexpr (GemmShape<BN>::kClusterOk)
    e = cudaFuncSetAttribute(gemm_tc_kernel<BN, EPI, kTcCluster>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_tc_kernel<BN, EPI, kTcWhole>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_tc_kernel<BN, EPI, kTcScratch>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             bytes);
  return e;
}

template <int BN>
static cudaError_t set_attr_bn() {
  cudaError_t e;
  if ((e = set_attr_one<BN, kEpiStoreF16>()) != cudaSuccess) return e;
  if ((e = set_attr_one<BN, kEpiResidF32>()) != cudaSuccess) return e;
  if ((e = set_attr_one<BN, kEpiSwiGLU>()) != cudaSuccess) return e;
  if ((e = set_attr_one<BN, kEpiArgmax>()) != cudaSuccess) return e;
  if constexpr (BN <= 64) e = set_attr_one<BN, kEpiQKV>();
  return e;
}

cudaError_t gemm_init_attributes() {
  cudaError_t e;
  if ((e = set_attr_bn<32>()) != cudaSuccess) return e;
  if ((e = set_attr_bn<64>()) != cudaSuccess) return e;
  if ((e = set_attr_bn<128>()) != cudaSuccess) return e;
  if ((e = set_attr_bn<256>()) != cudaSuccess) return e;
  return gemm_wide_init_attributes();
}

}  // namespace gs
