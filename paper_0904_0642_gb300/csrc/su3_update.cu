// su3_update.cu -- the float update phases of one chain, and the choice
// between float and FP64 forms.
#include "su3_phase.cuh"

namespace su3g {

constexpr int kSubVariant = 3;  // the FP32 variant of a divided chain

// One switch for launching and for occupancy queries of the float forms:
// OP<S, V, WT, SUB, TOR>.
template <template <class, int, bool, bool, bool> class OP, bool WT, class... A>
static cudaError_t update_dispatch(int storage, int variant, bool sub, bool torus, A... a) {
  constexpr bool kT = !WT;
  const bool tor = torus && !WT;
  if (variant == kFloatLanes && !WT) {
    if (storage == 2)
      return sub ? OP<StoreF32x18, kLanesVariant, false, true, false>::run(a...)
                 : OP<StoreF32x18, kLanesVariant, false, false, false>::run(a...);
    return sub ? OP<StoreF32x12, kLanesVariant, false, true, false>::run(a...)
               : OP<StoreF32x12, kLanesVariant, false, false, false>::run(a...);
  }
  // (links read before the wait come from L2: the coherent store forms)
  if (variant == kFloatEarly && tor)
    return storage == 2 ? OP<StoreF32x18T<true>, kEarlyVariant, false, false, kT>::run(a...)
                        : OP<StoreF32x12T<true>, kEarlyVariant, false, false, kT>::run(a...);
  if (variant == kFloatParked1 && storage == 1 && !WT && !sub)
    return tor ? OP<StoreF32x12, kParked1, false, false, kT>::run(a...) : OP<StoreF32x12, kParked1, false, false, false>::run(a...);
  if (variant == kFloatParked0 && !WT && !sub) {
    if (storage == 2)
      return tor ? OP<StoreF32x18, kParked0, false, false, kT>::run(a...) : OP<StoreF32x18, kParked0, false, false, false>::run(a...);
    return tor ? OP<StoreF32x12, kParked0, false, false, kT>::run(a...) : OP<StoreF32x12, kParked0, false, false, false>::run(a...);
  }
  if (variant >= kFloatEarly && !WT) {
    if (storage == 2)
      return sub ? OP<StoreF32x18T<true>, kEarlyRolled, false, true, false>::run(a...)
                 : OP<StoreF32x18T<true>, kEarlyRolled, false, false, false>::run(a...);
    return sub ? OP<StoreF32x12T<true>, kEarlyRolled, false, true, false>::run(a...)
               : OP<StoreF32x12T<true>, kEarlyRolled, false, false, false>::run(a...);
  }
  if (storage == 2) {
    if (sub) return OP<StoreF32x18, kSubVariant, WT, true, false>::run(a...);
    return tor ? OP<StoreF32x18, 0, false, false, kT>::run(a...) : OP<StoreF32x18, 0, WT, false, false>::run(a...);
  }
  if (sub) return OP<StoreF32x12, kSubVariant, WT, true, false>::run(a...);
  switch (variant) {
    case 0: return tor ? OP<StoreF32x12, 0, false, false, kT>::run(a...) : OP<StoreF32x12, 0, WT, false, false>::run(a...);
    case 1: return tor ? OP<StoreF32x12, 1, false, false, kT>::run(a...) : OP<StoreF32x12, 1, WT, false, false>::run(a...);
    case 2: return OP<StoreF32x12, 2, WT, false, false>::run(a...);
    case 3: return OP<StoreF32x12, 3, WT, false, false>::run(a...);
    default: return OP<StoreF32x12, 4, WT, false, false>::run(a...);
  }
}

cudaError_t launch_update(int storage, int variant, bool weighted, bool sub, bool torus, const ChainDesc &d,
                          ChainCtl *ctl, const UpdateStep &step, int grid, int block, cudaStream_t st, bool pdl) {
  if (storage == 0) return launch_update64(variant, weighted, sub, d, ctl, step, grid, block, st, pdl);
  if (sub && variant < kFloatLanes) variant = kSubVariant;
  if (block > tick_max_threads(storage, variant)) return cudaErrorInvalidConfiguration;
  const ChainDesc *pd = &d;
  const UpdateStep *pu = &step;
  return weighted ? update_dispatch<UpdateLaunch, true>(storage, variant, sub, torus, pd, ctl, pu, grid, block, st, pdl)
                  : update_dispatch<UpdateLaunch, false>(storage, variant, sub, torus, pd, ctl, pu, grid, block, st, pdl);
}

cudaError_t update_occupancy(int storage, int variant, bool weighted, bool sub, bool torus, int block,
                             int *ctas_per_sm) {
  *ctas_per_sm = 0;
  if (storage == 0) return update_occupancy64(variant, weighted, sub, block, ctas_per_sm);
  if (sub && variant < kFloatLanes) variant = kSubVariant;
  if (block > tick_max_threads(storage, variant)) return cudaSuccess;
  return weighted ? update_dispatch<UpdateOccupancy, true>(storage, variant, sub, torus, block, ctas_per_sm)
                  : update_dispatch<UpdateOccupancy, false>(storage, variant, sub, torus, block, ctas_per_sm);
}

// f(kernel) with the float k_sweeps form of a storage.
template <class F>
static auto by_sweeps(int storage, bool sub, F &&f) {
  if (storage == 2) return sub ? f(k_sweeps<StoreF32x18T<true>, true>) : f(k_sweeps<StoreF32x18T<true>, false>);
  return sub ? f(k_sweeps<StoreF32x12T<true>, true>) : f(k_sweeps<StoreF32x12T<true>, false>);
}

bool sweeps_supported(int storage, bool sub) {
  if (storage == 0) return sweeps_supported64(sub);
  return by_sweeps(storage, sub, [](auto *k) { return cluster_ctas(k, kClusterThreads); }) > 0;
}

cudaError_t launch_sweeps(int storage, bool sub, const ChainDesc &d, ChainCtl *ctl, int sweeps, cudaStream_t st,
                          bool pdl) {
  if (storage == 0) return launch_sweeps64(sub, d, ctl, sweeps, st, pdl);
  return by_sweeps(storage, sub, [&](auto *k) { return launch_cluster(k, d, ctl, sweeps, st, pdl); });
}

cudaError_t bounds_record_update(unsigned long long out[3]) {
  out[0] = out[1] = out[2] = 0;
#ifdef SU3_DEBUG_BOUNDS
  return cudaMemcpyFromSymbol(out, g_bounds, 3 * sizeof(unsigned long long));
#else
  return cudaSuccess;
#endif
}

}  // namespace su3g
