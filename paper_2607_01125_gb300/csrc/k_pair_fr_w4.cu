// Instantiations of the few-row pair forward for INT4 (g128) weights with bf16 activations.
#include "pair_fr_kernel.cuh"

namespace zoact {
namespace pairfr {

template <bool GATED>
static int launch_one(Ctx* ctx, const TmaSet& tm, const Params& p, const FrArgs& fr, int smem) {
  auto kern = pair_fr_kernel<__nv_bfloat16, GATED, true>;
  // (the most a plan may take: another thread's call never lowers it between this and the launch)
  ZOACT_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, CTA_SMEM));
  const unsigned tiles = (unsigned)((p.d_out + WR - 1) / WR);
  ZOACT_CUDA_TRY(launch_pdl_cluster(ctx, kern, dim3(tiles * fr.splits), dim3(fr_threads(true)), (size_t)smem,
                                    (unsigned)fr.splits, tm, p, fr));
  ++ctx->n_launch;
  ZOACT_CHECK_LAUNCH();
  return ZOACT_OK;
}

int dispatch_fr_w4(Ctx* ctx, bool gated, const TmaSet& tm, const Params& p, const FrArgs& fr, int smem) {
  return gated ? launch_one<true>(ctx, tm, p, fr, smem) : launch_one<false>(ctx, tm, p, fr, smem);
}

}  // namespace pairfr
}  // namespace zoact
