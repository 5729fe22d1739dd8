// su3_update64.cu -- the FP64 update phases of one chain.
#include "su3_phase.cuh"

namespace su3g {

template <template <class, int, bool, bool, bool> class OP, class... A>
static cudaError_t update_dispatch64(int variant, bool weighted, bool sub, A... a) {
  if (weighted)
    return sub ? OP<StoreF64x18, 10, true, true, false>::run(a...) : OP<StoreF64x18, 10, true, false, false>::run(a...);
  if (variant == 1)
    return sub ? OP<StoreF64x18, kCoopVariant, false, true, false>::run(a...)
               : OP<StoreF64x18, kCoopVariant, false, false, false>::run(a...);
  return sub ? OP<StoreF64x18, 10, false, true, false>::run(a...) : OP<StoreF64x18, 10, false, false, false>::run(a...);
}

cudaError_t launch_update64(int variant, bool weighted, bool sub, const ChainDesc &d, ChainCtl *ctl,
                            const UpdateStep &step, int grid, int block, cudaStream_t st, bool pdl) {
  if (block > tick_max_threads(0, variant)) return cudaErrorInvalidConfiguration;
  return update_dispatch64<UpdateLaunch>(variant, weighted, sub, &d, ctl, &step, grid, block, st, pdl);
}

cudaError_t update_occupancy64(int variant, bool weighted, bool sub, int block, int *ctas_per_sm) {
  if (block > tick_max_threads(0, variant)) return cudaSuccess;
  return update_dispatch64<UpdateOccupancy>(variant, weighted, sub, block, ctas_per_sm);
}

bool sweeps_supported64(bool sub) {
  return (sub ? cluster_ctas(k_sweeps<StoreF64x18T<true>, true>, kClusterThreads)
              : cluster_ctas(k_sweeps<StoreF64x18T<true>, false>, kClusterThreads)) > 0;
}

cudaError_t launch_sweeps64(bool sub, const ChainDesc &d, ChainCtl *ctl, int sweeps, cudaStream_t st, bool pdl) {
  return sub ? launch_cluster(k_sweeps<StoreF64x18T<true>, true>, d, ctl, sweeps, st, pdl)
             : launch_cluster(k_sweeps<StoreF64x18T<true>, false>, d, ctl, sweeps, st, pdl);
}

cudaError_t bounds_record_update64(unsigned long long out[3]) {
  out[0] = out[1] = out[2] = 0;
#ifdef SU3_DEBUG_BOUNDS
  return cudaMemcpyFromSymbol(out, g_bounds, 3 * sizeof(unsigned long long));
#else
  return cudaSuccess;
#endif
}

}  // namespace su3g
