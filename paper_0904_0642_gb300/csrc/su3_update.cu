// su3_update.cu -- kernels of one chain (sm_103a): the update phases, the
// re-unitarisation and the measurement of a lattice whose schedule the host
// knows.  The descriptor is a kernel parameter: geometry and pointers are
// uniform values from the constant bank, nothing is loaded before the links.
#include "su3_launch.h"
#include "su3_site.cuh"

namespace su3g {

// Every kernel may be scheduled before the previous one of the stream has
// finished (programmatic launch): wait for its completion and memory before
// touching anything, then let the next kernel be scheduled.  Both are no-ops
// for an ordinary launch.
__device__ __forceinline__ void wait_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The sweep counter of a schedule's launch (its first one copies it).
__device__ __forceinline__ uint32_t next_base(ChainCtl *ctl, const UpdateStep &u) {
  const uint32_t base = __ldcg(u.first ? &ctl->nxt : &ctl->cur);
  if (u.first && blockIdx.x == 0 && threadIdx.x == 0) ctl->cur = base;
  return base;
}

template <class S, int V, bool WT, bool SUB, bool TOR>
__global__ void __launch_bounds__(TickBounds<V>::kThreads, TickBounds<V>::kMinBlocks)
    k_update(const __grid_constant__ ChainDesc d, ChainCtl *ctl, const UpdateStep u) {
  uint32_t np = 0, na = 0;
  if constexpr (kLanesOf<V> > 1) {
    // The site and the draws need no link: they run before the wait, while the
    // previous phase ends - except in a schedule's first two launches, whose
    // predecessors may still be writing the sweep counter.
    uint32_t base = 0;
    const bool early = u.early != 0;
    if (early) base = __ldcg(&ctl->cur);
    WarpLinks<S, SUB> w;
    int lt = blockIdx.x;
    WarpPlace p = warp_place<kCoopLanes>(d, lt);
    if (early && p.jw < d.Vn) w.prepare(d, base + u.offset, u.colour, u.mu, p.layer, p.jw);
    wait_previous();
    if (!early) base = next_base(ctl, u);
    if (u.advance && blockIdx.x == 0 && threadIdx.x == 0) ctl->nxt = base + u.advance;
    if (!early && p.jw < d.Vn) w.prepare(d, base + u.offset, u.colour, u.mu, p.layer, p.jw);
    while (true) {
      if (p.jw < d.Vn) w.template update<false>(d, base + u.offset, u.colour, u.mu, p.slot, np, na);
      lt += gridDim.x;
      if (lt >= u.tiles) break;
      p = warp_place<kCoopLanes>(d, lt);
      if (p.jw < d.Vn) w.prepare(d, base + u.offset, u.colour, u.mu, p.layer, p.jw);
    }
  } else if constexpr (kIsEarly<V> || kIsParked<V>) {
    // A launch that leaves room on the GPU runs beside its predecessor: all
    // but what depends on that one comes before the wait.  The previous
    // launch writes links of direction prev only, so the draws, and the sums
    // over the staples up to those of direction prev, do not wait (in the
    // sums' order: three of the four directions of a 4-D sweep gain).  The
    // launch before that has ended: every CTA of the previous one waited for
    // it.  Links come from L2: only the wait makes L1 forget what this SM
    // read before earlier launches wrote.  The parked forms have only the
    // draws before the wait and read links as ever.
    bool waited = u.early == 0;
    uint32_t base;
    if (waited) {
      wait_previous();
      base = next_base(ctl, u);
    } else {
      base = __ldcg(&ctl->cur);
    }
    const int prev = u.mu == 0 ? d.D - 1 : u.mu - 1;
    const auto ready = [&](int nu) {
      if (!waited && (kIsParked<V> || nu == prev)) {
        wait_previous();
        waited = true;
      }
    };
    for (int lt = blockIdx.x; lt < u.tiles; lt += gridDim.x)
      update_tile<S, V, WT, SUB, TOR>(d, base + u.offset, u.colour, u.mu, lt, np, na, ready);
    ready(prev);  // a thread without a link
    if (u.advance && blockIdx.x == 0 && threadIdx.x == 0) ctl->nxt = base + u.advance;
  } else {
    wait_previous();
    const uint32_t base = next_base(ctl, u);
    if (u.advance && blockIdx.x == 0 && threadIdx.x == 0) ctl->nxt = base + u.advance;
    for (int lt = blockIdx.x; lt < u.tiles; lt += gridDim.x)
      update_tile<S, V, WT, SUB, TOR>(d, base + u.offset, u.colour, u.mu, lt, np, na);
  }
  flush_counters(d, np, na);
}

// Whole sweeps of a small lattice in one launch of one thread-block cluster
// (eight lanes per link): the phases are separated by the cluster's hardware
// barrier instead of a kernel boundary, and the code stays in the instruction
// caches.  Links are read through L2 (COH): other CTAs have written them.
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <class S, bool SUB>
__global__ void __launch_bounds__(kClusterThreads, 1)
    k_sweeps(const __grid_constant__ ChainDesc d, ChainCtl *ctl, int sweeps) {
  wait_previous();
  const uint32_t base = __ldcg(&ctl->nxt);
  constexpr int kPerWarp = 32 / kCoopLanes;
  const int per_vl = (d.Vn + kPerWarp - 1) / kPerWarp, warps = d.nlayers * d.nb * per_vl;
  const int w0 = (int)(blockIdx.x * blockDim.x + threadIdx.x) / 32, nw = (int)(gridDim.x * blockDim.x) / 32;
  uint32_t np = 0, na = 0;
#pragma unroll 1
  for (int i = 0; i < sweeps * 2 * d.D; ++i) {
    const int s = i / (2 * d.D), st = i - s * 2 * d.D;
    const int colour = st >= d.D ? 1 : 0, mu = st - colour * d.D;
    int w = w0;
#pragma unroll 1
    do {
      const int vl = w / per_vl, j0 = (w - vl * per_vl) * kPerWarp;
      WarpLinks<S, SUB> links;
      // the site and the draws need no link: the first of a phase before the
      // wait for the previous phase's links
      if (w < warps) links.prepare(d, base + (uint32_t)s, colour, mu, vl, j0);
      if (i > 0 && w == w0) cluster_wait();
      if (w < warps) links.template update<true>(d, base + (uint32_t)s, colour, mu, w, np, na);
      w += nw;
    } while (w < warps);
    cluster_arrive();
  }
  cluster_wait();
  flush_counters(d, np, na);
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl->nxt = base + (uint32_t)sweeps;
}

// One thread per link: blockIdx.z = colour D + mu, blockIdx.y a (virtual) layer.
template <class S, bool SUB>
__global__ void __launch_bounds__(128) k_reunit(const __grid_constant__ ChainDesc d) {
  wait_previous();
  const int jj = blockIdx.x * blockDim.x + threadIdx.x;
  if (jj >= d.Vn) return;
  const int colour = (int)blockIdx.z / d.D, mu = (int)blockIdx.z - colour * d.D;
  const int js = SUB ? (site_of<true>(d, blockIdx.y, colour, jj).s >> 1) : jj;
  reunit_link<S>(plane_ptr<S>(d, blockIdx.y, colour, mu), d.Vh, js);
}

// Plaquettes and Polyakov lines (one per thread) of layer blockIdx.y, the
// lines first: the longest work starts first.  Plaquettes: FP64 one plane of a
// site per thread; FP32 all planes of a site (SPLIT false), or eight lanes
// per site (SPLIT: lattices that do not fill the GPU with a site per thread).
// The last CTA to finish sums the CTAs' partial sums in a fixed order.
template <class S, bool SUB, bool SPLIT>
__global__ void __launch_bounds__(128, sizeof(typename S::R) == 8 ? 3 : 5) k_measure(const __grid_constant__ ChainDesc d, double *out, ChainCtl *ctl,
                                                 int record) {
  __shared__ double s_red[32];
  __shared__ double s_sum[3][kPartVals];
  __shared__ int s_last;
  wait_previous();
  const int layer = blockIdx.y, T = d.D - 1;
  constexpr bool kFixed = std::is_same<S, StoreF64x18>::value;
  constexpr int kSites = SPLIT ? 16 : 128;  // sites of a tile
  const int nl = (SUB && d.hpad[T]) ? 0 : d.Vn / d.idims[T];  // lines per colour of a box
  const int planes = kFixed ? d.D * T / 2 : 1;
  const int ltiles = (nl + 127) / 128, stiles = (d.Vn + kSites - 1) / kSites, nlt = d.nb * 2 * ltiles;
  double v[kPartVals] = {0, 0, 0, 0};
  for (int t = blockIdx.x; t < nlt + d.nb * 2 * stiles * planes; t += gridDim.x) {
    if (t < nlt) {
      const int cb = t / ltiles, jj = (t - cb * ltiles) * 128 + threadIdx.x, colour = cb & 1;
      if (jj >= nl) continue;
      const SiteGeo g = site_of<SUB>(d, layer * d.nb + (cb >> 1), colour, jj);
      const C<double> p = line_trace<S, SUB>(d, g, colour, jj);
      v[2] += p.re;
      v[3] += p.im;
      continue;
    }
    const int r = t - nlt, pc = r / stiles, cb = pc / planes, colour = cb & 1, vl = layer * d.nb + (cb >> 1);
    if constexpr (SPLIT) {
      const int jj = (r - pc * stiles) * kSites + (threadIdx.x >> 3);
      typename S::R ps, pt;
      site_plaquettes_split<S, SUB>(d, site_of<SUB>(d, vl, colour, min(jj, d.Vn - 1)), colour, ps, pt);
      if ((threadIdx.x & 7) == 0 && jj < d.Vn) {
        v[0] += to_double(ps);
        v[1] += to_double(pt);
      }
    } else {
      const int jj = (r - pc * stiles) * kSites + threadIdx.x;
      if (jj >= d.Vn) continue;
      const SiteGeo g = site_of<SUB>(d, vl, colour, jj);
      if constexpr (kFixed) {
        int nu = 1, mu = pc - cb * planes;  // planes (0,1), (0,2), (1,2), (0,3), ...
        while (mu >= nu) mu -= nu++;
        PlaquetteSum p;
        add_plaquette<SUB>(d, g, colour, jj, mu, nu, p);
        v[0] += nu == T ? 0.0 : p.value();
        v[1] += nu == T ? p.value() : 0.0;
      } else {
        typename S::R ps, pt;
        site_plaquettes<S, SUB>(d, g, colour, ps, pt);
        v[0] += to_double(ps);
        v[1] += to_double(pt);
      }
    }
  }
  block_reduce(v, s_red);
  if (threadIdx.x == 0) {
    const int slot = layer * gridDim.x + blockIdx.x;
    if (in_bounds(slot, d.nlayers * kMeasureCtas, kBoundsPartial))
      for (int k = 0; k < kPartVals; ++k) d.partials[(size_t)slot * kPartVals + k] = v[k];
    __threadfence();
    s_last = atomicAdd(&ctl->done, 1u) == gridDim.x * gridDim.y - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const uint32_t slot = ctl->n_meas;
  if (record) out = d.results + (size_t)(slot % (uint32_t)d.result_cap) * (d.nlayers + 1) * kMeasVals;
  for (int l = 0; l < d.nlayers; ++l) {
    double w[kPartVals] = {0, 0, 0, 0};
    for (int b = threadIdx.x; b < gridDim.x; b += 128)
#pragma unroll
      for (int k = 0; k < kPartVals; ++k) w[k] += __ldcg(d.partials + (size_t)(l * gridDim.x + b) * kPartVals + k);
    block_reduce(w, s_red);
    if (threadIdx.x == 0)
#pragma unroll
      for (int k = 0; k < kPartVals; ++k) {
        s_sum[l][k] = w[k];
        s_sum[d.nlayers][k] = l == 0 ? w[k] : s_sum[d.nlayers][k] + w[k];
      }
  }
  __syncthreads();
  // one value per thread: the divisions side by side
  if (threadIdx.x < (d.nlayers + 1) * kMeasVals) {
    const int l = threadIdx.x / kMeasVals;
    out[threadIdx.x] = measured_value(d, s_sum[l], l == d.nlayers ? (double)l : 1.0, threadIdx.x - l * kMeasVals);
  }
  if (threadIdx.x == 0) ctl->done = 0;
  if (!record) return;
  // a chain whose links were replaced restarts its action bookkeeping here
  const int anchor = ctl->anchor;
  __syncthreads();
  if (anchor) {
    for (int i = threadIdx.x; i < (d.nlayers + 1) * kMeasVals; i += 128) d.ref_meas[i] = out[i];
    for (int i = threadIdx.x; i < d.n_action_slots; i += 128) d.action_slots[i] = 0.0;
  }
  if (threadIdx.x == 0) {
    ctl->n_meas = slot + 1;
    ctl->anchor = 0;
  }
}

__global__ void k_set_ctl(ChainCtl *ctl, uint32_t sweep, uint32_t n_meas, int anchor) {
  *ctl = ChainCtl{sweep, sweep, n_meas, anchor, 0u, {0, 0, 0}};
}

// ------------------------------------------------------------------ launchers

constexpr int kSubVariant = 3;  // the FP32 variant of a divided chain

// Dynamic shared memory per thread.
template <int V>
constexpr int kSharedOf = kIsParked<V> ? kParkedBytes : 0;

template <class S, int V, bool WT, bool SUB, bool TOR>
struct UpdateLaunch {
  static cudaError_t run(const ChainDesc *d, ChainCtl *ctl, const UpdateStep *u, int grid, int block, cudaStream_t st,
                         bool pdl) {
    return launch_shared(k_update<S, V, WT, SUB, TOR>, dim3((unsigned)grid), block, kSharedOf<V> * block, st, pdl, *d,
                         ctl, *u);
  }
};
template <class S, int V, bool WT, bool SUB, bool TOR>
struct UpdateOccupancy {
  static cudaError_t run(int block, int *ctas) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, k_update<S, V, WT, SUB, TOR>, block,
                                                         kSharedOf<V> * block);
  }
};

// One switch for launching and for occupancy queries: OP<S, V, WT, SUB, TOR>.
template <template <class, int, bool, bool, bool> class OP, bool WT, class... A>
static cudaError_t update_dispatch(int storage, int variant, bool sub, bool torus, A... a) {
  constexpr bool kT = !WT;
  const bool tor = torus && !WT;
  if (storage == 0) {
    if (variant == 1 && !WT)
      return sub ? OP<StoreF64x18, kCoopVariant, false, true, false>::run(a...)
                 : OP<StoreF64x18, kCoopVariant, false, false, false>::run(a...);
    return sub ? OP<StoreF64x18, 10, WT, true, false>::run(a...) : OP<StoreF64x18, 10, WT, false, false>::run(a...);
  }
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
  if (sub && storage != 0 && variant < kFloatLanes) variant = kSubVariant;
  if (block > tick_max_threads(storage, variant)) return cudaErrorInvalidConfiguration;
  const ChainDesc *pd = &d;
  const UpdateStep *pu = &step;
  return weighted ? update_dispatch<UpdateLaunch, true>(storage, variant, sub, torus, pd, ctl, pu, grid, block, st, pdl)
                  : update_dispatch<UpdateLaunch, false>(storage, variant, sub, torus, pd, ctl, pu, grid, block, st, pdl);
}

cudaError_t update_occupancy(int storage, int variant, bool weighted, bool sub, bool torus, int block,
                             int *ctas_per_sm) {
  *ctas_per_sm = 0;
  if (sub && storage != 0 && variant < kFloatLanes) variant = kSubVariant;
  if (block > tick_max_threads(storage, variant)) return cudaSuccess;
  return weighted ? update_dispatch<UpdateOccupancy, true>(storage, variant, sub, torus, block, ctas_per_sm)
                  : update_dispatch<UpdateOccupancy, false>(storage, variant, sub, torus, block, ctas_per_sm);
}

// The largest cluster the device takes for k_sweeps (0: none).
template <class K>
static int cluster_ctas(K *kernel, int threads) {
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kClusterCtas);
  cfg.blockDim = dim3((unsigned)threads);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim = {kClusterCtas, 1, 1};
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n > 0 ? kClusterCtas : 0;
}

// f(kernel) with the k_sweeps form of a storage.
template <class F>
static auto by_sweeps(int storage, bool sub, F &&f) {
  if (storage == 0) return sub ? f(k_sweeps<StoreF64x18T<true>, true>) : f(k_sweeps<StoreF64x18T<true>, false>);
  if (storage == 2) return sub ? f(k_sweeps<StoreF32x18T<true>, true>) : f(k_sweeps<StoreF32x18T<true>, false>);
  return sub ? f(k_sweeps<StoreF32x12T<true>, true>) : f(k_sweeps<StoreF32x12T<true>, false>);
}

bool sweeps_supported(int storage, bool sub) {
  return by_sweeps(storage, sub, [](auto *k) { return cluster_ctas(k, kClusterThreads); }) > 0;
}

cudaError_t launch_sweeps(int storage, bool sub, const ChainDesc &d, ChainCtl *ctl, int sweeps, cudaStream_t st,
                          bool pdl) {
  // as many threads as the links need lanes (whole warps), up to the limit
  const int warps = d.nlayers * d.nb * ((d.Vn + 3) / 4);
  const int per = (warps + kClusterCtas - 1) / kClusterCtas;
  const int threads = 32 * (per < kClusterThreads / 32 ? per : kClusterThreads / 32);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kClusterCtas);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim = {kClusterCtas, 1, 1};
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return by_sweeps(storage, sub, [&](auto *k) { return cudaLaunchKernelEx(&cfg, k, d, ctl, sweeps); });
}

cudaError_t launch_reunit(int storage, bool sub, const ChainDesc &d, cudaStream_t st, bool pdl) {
  const dim3 grid((unsigned)((d.Vn + 127) / 128), (unsigned)(d.nlayers * d.nb), (unsigned)(2 * d.D));
  return by_storage(storage, [&](auto s) {
    using S = decltype(s);
    return sub ? launch_ex(k_reunit<S, true>, grid, 128, st, pdl, d) : launch_ex(k_reunit<S, false>, grid, 128, st, pdl, d);
  });
}

cudaError_t launch_measure(int storage, bool sub, const ChainDesc &d, double *out, ChainCtl *ctl, cudaStream_t st,
                           bool pdl) {
  const int T = d.D - 1, nl = (sub && d.hpad[T]) ? 0 : d.Vn / d.idims[T];
  const int planes = storage == 0 ? d.D * T / 2 : 1;
  const bool split = storage != 0 && (long long)d.nlayers * d.nb * d.Vn <= kSplitSites;
  const int sites = split ? 16 : 128, most = storage == 0 ? kMeasureCtasF64 : kMeasureCtas;
  const long long tiles = (long long)d.nb * 2 * ((nl + 127) / 128 + (long long)planes * ((d.Vn + sites - 1) / sites));
  const dim3 grid((unsigned)(tiles < most ? tiles : most), (unsigned)d.nlayers);
  const int record = out ? 0 : 1;
  return by_storage(storage, [&](auto s) {
    using S = decltype(s);
    if constexpr (!std::is_same<S, StoreF64x18>::value)
      if (split)
        return sub ? launch_ex(k_measure<S, true, true>, grid, 128, st, pdl, d, out, ctl, record)
                   : launch_ex(k_measure<S, false, true>, grid, 128, st, pdl, d, out, ctl, record);
    return sub ? launch_ex(k_measure<S, true, false>, grid, 128, st, pdl, d, out, ctl, record)
               : launch_ex(k_measure<S, false, false>, grid, 128, st, pdl, d, out, ctl, record);
  });
}

cudaError_t launch_set_ctl(ChainCtl *ctl, uint32_t sweep, uint32_t n_meas, int anchor, cudaStream_t st) {
  k_set_ctl<<<1, 1, 0, st>>>(ctl, sweep, n_meas, anchor);
  return cudaGetLastError();
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
