// su3_phase.cuh -- the update kernels of one chain (sm_103a), whose schedule
// the host knows.  The descriptor is a kernel parameter: geometry and pointers
// are uniform values from the constant bank, nothing is loaded before the
// links.  The float forms are compiled in su3_update.cu, the FP64 forms in
// su3_update64.cu, re-unitarisation and measurement in su3_stages.cu, the fused
// stage machine of many chains in su3_tick.cu: a module is loaded by a process
// at the first use of one of its kernels, and the update forms together take
// 25 ms to load.
#pragma once
#include "su3_launch.h"
#include "su3_site.cuh"

namespace su3g {

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

// ------------------------------------------------------------------ launching

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

// The largest cluster the device takes for k_sweeps (0: none).
template <class K>
static inline int cluster_ctas(K *kernel, int threads) {
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

// Launch a form of k_sweeps: as many threads as the links need lanes (whole
// warps), up to the limit.
template <class K>
static inline cudaError_t launch_cluster(K *kernel, const ChainDesc &d, ChainCtl *ctl, int sweeps, cudaStream_t st,
                                         bool pdl) {
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
  return cudaLaunchKernelEx(&cfg, kernel, d, ctl, sweeps);
}

}  // namespace su3g
