// Instantiations of the few-row pair forward for bf16 weights and activations.
#include "pair_fr_kernel.cuh"

namespace zoact {
namespace pairfr {

template <bool GATED>
static int launch_one(Ctx* ctx, const TmaSet& tm, const Params& p, const FrArgs& fr, int smem) {
  auto kern = pair_fr_kernel<__nv_bfloat16, GATED, false>;
  // (the most a plan may take: another thread's call never lowers it between this and the launch)
  ZOACT_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, CTA_SMEM));
  const unsigned tiles = (unsigned)((p.d_out + WR - 1) / WR);
  ZOACT_CUDA_TRY(launch_pdl_cluster(ctx, kern, dim3(tiles * fr.splits), dim3(fr_threads(false)), (size_t)smem,
                                    (unsigned)fr.splits, tm, p, fr));
  ++ctx->n_launch;
  ZOACT_CHECK_LAUNCH();
  return ZOACT_OK;
}

// Clusters of `size` CTAs with smem bytes each that the device runs at once (at least 1; the whole family is alike).
int fr_max_clusters(int size, int smem) {
  auto kern = pair_fr_kernel<__nv_bfloat16, false, false>;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)size;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)size);
  cfg.blockDim = dim3(fr_threads(false));
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, CTA_SMEM) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 1;
  }
  return n > 1 ? n : 1;
}

int dispatch_fr_bf16(Ctx* ctx, bool gated, const TmaSet& tm, const Params& p, const FrArgs& fr, int smem) {
  return gated ? launch_one<true>(ctx, tm, p, fr, smem) : launch_one<false>(ctx, tm, p, fr, smem);
}

}  // namespace pairfr
}  // namespace zoact
