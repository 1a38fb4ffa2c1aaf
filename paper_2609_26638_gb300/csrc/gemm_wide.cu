// gemm_wide.cu -- instantiations and launcher of the persistent GEMM.
#include "gemm_wide.cuh"
#include "internal.h"

namespace gs {

template <int BN, int EPI>
static cudaError_t launch_one(const CUtensorMap& tmW, const CUtensorMap& tmX, GemmArgs a,
                              int feat_tiles, int tok_tiles, cudaStream_t s, bool pdl) {
  using S = WideShape<BN>;
  a.tok_tiles = tok_tiles;
  // the LM head of a small window: more tiles than SMs and one token tile
  if constexpr (BN == 32 && EPI == kEpiArgmax) {
    if (tok_tiles == 1 && feat_tiles > kNumSMs && S::resident_stages(EPI, a.K / 64) > 0)
      return launch_ex(gemm_wide_kernel<BN, EPI, true>, dim3(feat_tiles), dim3(S::kThreads),
                       S::smem_bytes(EPI), s, pdl, dim3(1, 1, 1), tmW, tmX, a);
  }
  return launch_ex(gemm_wide_kernel<BN, EPI, false>, dim3(feat_tiles * tok_tiles), dim3(S::kThreads), S::smem_bytes(EPI), s,
                   pdl, dim3(1, 1, 1), tmW, tmX, a);
}

template <int BN>
static cudaError_t launch_bn(int epi, const CUtensorMap& tmW, const CUtensorMap& tmX,
                             const GemmArgs& a, int ft, int tt, cudaStream_t s, bool pdl) {
  switch (epi) {
    case kEpiStoreF16: return launch_one<BN, kEpiStoreF16>(tmW, tmX, a, ft, tt, s, pdl);
    case kEpiResidF32: return launch_one<BN, kEpiResidF32>(tmW, tmX, a, ft, tt, s, pdl);
    case kEpiSwiGLU: return launch_one<BN, kEpiSwiGLU>(tmW, tmX, a, ft, tt, s, pdl);
    case kEpiArgmax: return launch_one<BN, kEpiArgmax>(tmW, tmX, a, ft, tt, s, pdl);
    case kEpiQKV: return launch_one<BN, kEpiQKV>(tmW, tmX, a, ft, tt, s, pdl);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_gemm_wide(int bn, int epi, const CUtensorMap& tmW, const CUtensorMap& tmX,
                             const GemmArgs& a, int ft, int tt, cudaStream_t s, bool pdl) {
  switch (bn) {
    case 32: return launch_bn<32>(epi, tmW, tmX, a, ft, tt, s, pdl);
    case 64: return launch_bn<64>(epi, tmW, tmX, a, ft, tt, s, pdl);
    case 96: return launch_bn<96>(epi, tmW, tmX, a, ft, tt, s, pdl);
    case 144: return launch_bn<144>(epi, tmW, tmX, a, ft, tt, s, pdl);
    case 192: return launch_bn<192>(epi, tmW, tmX, a, ft, tt, s, pdl);
    case 256: return launch_bn<256>(epi, tmW, tmX, a, ft, tt, s, pdl);
  }
  return cudaErrorInvalidValue;
}

template <int BN, int EPI>
static cudaError_t set_one() {
  if constexpr (BN == 32 && EPI == kEpiArgmax) {
    const cudaError_t e =
        cudaFuncSetAttribute(gemm_wide_kernel<BN, EPI, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             WideShape<BN>::smem_bytes(EPI));
    if (e != cudaSuccess) return e;
  }
  return cudaFuncSetAttribute(gemm_wide_kernel<BN, EPI, false>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              WideShape<BN>::smem_bytes(EPI));
}

template <int BN>
static cudaError_t set_bn() {
  cudaError_t e;
  if ((e = set_one<BN, kEpiStoreF16>()) != cudaSuccess) return e;
  if ((e = set_one<BN, kEpiResidF32>()) != cudaSuccess) return e;
  if ((e = set_one<BN, kEpiSwiGLU>()) != cudaSuccess) return e;
  if ((e = set_one<BN, kEpiArgmax>()) != cudaSuccess) return e;
  return set_one<BN, kEpiQKV>();
}

cudaError_t gemm_wide_init_attributes() {
  cudaError_t e;
  if ((e = set_bn<32>()) != cudaSuccess) return e;
  if ((e = set_bn<64>()) != cudaSuccess) return e;
  if ((e = set_bn<96>()) != cudaSuccess) return e;
  if ((e = set_bn<144>()) != cudaSuccess) return e;
  if ((e = set_bn<192>()) != cudaSuccess) return e;
  return set_bn<256>();
}

}  // namespace gs
