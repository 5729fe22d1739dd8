// su3_tick.cu -- the fused stage machine of many chains (sm_103a).
//
// k_tick (engines of several chains, the server's): one persistent launch
//   advances every resident chain by one stage (a (colour, direction) update
//   phase, a re-unitarisation or a measurement).  One thread per site of the
//   tile (tile = CTA width); tiles of all chains are spread over a grid of
//   CTAs sized to the SM count.  The chains' stage machines advance at the end
//   of the launch (by the first warp to finish, into a second state slot, with
//   the last one flipping the slot parity; one resident chain: by the last
//   warp), and the last warp reduces measurement partial sums in a fixed
//   order.  An engine of one chain runs the kernels of su3_update.cu.
#include <type_traits>

#include "su3_launch.h"
#include "su3_site.cuh"

namespace su3g {

// ------------------------------------------------------------------ tick kernel

// Copy a chain's descriptor and its current state (of its two state slots,
// the one the launch's parity names; the parity is the same for the whole
// launch) into the CTA's shared memory.  Both slots and the parity are
// loaded together and the current one selected, so that no load waits for
// another.
__device__ __forceinline__ void load_chain(const EngineArgs &ea, int c, ChainDesc &sd, ChainState &ss, int &s_par) {
  const int n1 = sizeof(ChainDesc) / 4, n2 = sizeof(ChainState) / 4;
  const uint32_t *src1 = reinterpret_cast<const uint32_t *>(ea.desc + c);
  const uint32_t *src2 = reinterpret_cast<const uint32_t *>(ea.state + 2 * (size_t)c);
  uint32_t *dst1 = reinterpret_cast<uint32_t *>(&sd), *dst2 = reinterpret_cast<uint32_t *>(&ss);
  for (int i = threadIdx.x; i < n1; i += blockDim.x) dst1[i] = src1[i];
  for (int i = threadIdx.x; i < n2; i += blockDim.x) {
    const uint32_t w0 = __ldcg(src2 + i), w1 = __ldcg(src2 + n2 + i);
    const int par = __ldcg(&ea.hdr->parity);
    dst2[i] = par ? w1 : w0;
    if (i == 0) s_par = par;
  }
}

// The next chain of a CTA, staged in shared memory (multi-chain form).
struct ChainStaging {
  ChainDesc d;
  ChainState s;
};
struct NoStaging {};

// Start asynchronous copies (cp.async, one 4-byte word per thread at a
// time) of chain c's descriptor and current state into the CTA's staging
// buffer.  The CTA's next chain switch waits for them (cp.async.wait_all,
// then the barrier) and copies them over the current ones, instead of
// waiting behind that barrier for a round trip to L2.
__device__ __forceinline__ void stage_chain(const EngineArgs &ea, int c, int par, ChainStaging &stg) {
  const int n1 = sizeof(ChainDesc) / 4, n2 = sizeof(ChainState) / 4;
  const uint32_t *src1 = reinterpret_cast<const uint32_t *>(ea.desc + c);
  const uint32_t *src2 = reinterpret_cast<const uint32_t *>(ea.state + 2 * (size_t)c + par);
  uint32_t *dst1 = reinterpret_cast<uint32_t *>(&stg.d), *dst2 = reinterpret_cast<uint32_t *>(&stg.s);
  for (int i = threadIdx.x; i < n1 + n2; i += blockDim.x) {
    const uint32_t *src = i < n1 ? src1 + i : src2 + (i - n1);
    const unsigned dst = (unsigned)__cvta_generic_to_shared(i < n1 ? dst1 + i : dst2 + (i - n1));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// Copy the staged descriptor and state over the current ones (shared to
// shared, one word per thread at a time).
__device__ __forceinline__ void take_staged(ChainDesc &sd, ChainState &ss, const ChainStaging &stg) {
  const int n1 = sizeof(ChainDesc) / 4, n2 = sizeof(ChainState) / 4;
  const uint32_t *src1 = reinterpret_cast<const uint32_t *>(&stg.d), *src2 = reinterpret_cast<const uint32_t *>(&stg.s);
  uint32_t *dst1 = reinterpret_cast<uint32_t *>(&sd), *dst2 = reinterpret_cast<uint32_t *>(&ss);
  for (int i = threadIdx.x; i < n1 + n2; i += blockDim.x) {
    if (i < n1)
      dst1[i] = src1[i];
    else
      dst2[i - n1] = src2[i - n1];
  }
}

// Next stage of a chain's stage machine (the host keeps an identical mirror):
// the 2D update phases of a sweep, then a re-unitarisation and/or a
// measurement when the completed-sweep count is a multiple of their
// cadence; the chain goes idle when a sweep would start at its target.
struct StageParams {
  int D, reunit_every, measure_every;
};

__device__ __host__ inline void advance_stage(const StageParams &d, ChainState &s) {
  if (s.stage < 2 * d.D) {
    s.stage += 1;
    if (s.stage == 2 * d.D) {
      s.sweep += 1;
      const bool r = d.reunit_every > 0 && (s.sweep % (uint32_t)d.reunit_every) == 0;
      const bool m = d.measure_every > 0 && (s.sweep % (uint32_t)d.measure_every) == 0;
      s.stage = r ? kStageReunit : (m ? kStageMeasure : 0);
    }
  } else if (s.stage == kStageReunit) {
    const bool m = d.measure_every > 0 && (s.sweep % (uint32_t)d.measure_every) == 0;
    s.stage = m ? kStageMeasure : 0;
  } else {
    s.stage = 0;
  }
  if (s.stage == 0 && s.sweep >= s.target) s.active = 0;
}

__device__ __host__ inline void advance_stage(const ChainDesc &d, ChainState &s) {
  advance_stage(StageParams{d.D, d.reunit_every, d.measure_every}, s);
}

// The state of a chain after this launch's tick.
__device__ __forceinline__ ChainState next_state(const StageParams &p, ChainState s) {
  if (!s.active) return s;
  if (s.stage == kStageMeasure) {
    s.n_meas += 1;
    s.anchor = 0;  // the measurement restarts the bookkeeping if it was set
  }
  advance_stage(p, s);
  return s;
}

__device__ __forceinline__ bool measures(const ChainState &s) { return s.active && s.stage == kStageMeasure; }

// The end of a one-chain launch, by its last warp: finish the measurement
// and advance the chain's state in place (every other warp has read it).
__device__ __forceinline__ void finish_single_chain(const EngineArgs &ea, const ChainDesc &d, const ChainState &cs,
                                                    int par, int lane) {
  if (measures(cs)) {
    __threadfence();  // acquire the partials of every tile
    double *out = d.results + (size_t)(cs.n_meas % (uint32_t)d.result_cap) * (d.nlayers + 1) * kMeasVals;
    finalize_measure(d, d.partials, out);
    if (cs.anchor) restart_bookkeeping(d, out);
  }
  const ChainState st = next_state(StageParams{d.D, d.reunit_every, d.measure_every}, cs);
  if (lane == 0) {
    ea.state[par] = st;
    ea.hdr->done = 0u;
  }
}

// WT: compiled for engines holding a two-coupling DLT chain (any chain with
// beta1 != beta); unweighted chains compute identically in both forms.
// TOR: compiled for engines whose chains are all undivided periodic 4-D tori
// with one coupling and the default random-number key: the unrolled update
// with D, the layer and the site key fixed at compile time.  Its FP32 12-real
// variant 0 also stages the chain of the CTA's next tile in shared memory
// with cp.async while the current tile runs (tiles are dealt out in
// grid-stride order, so a CTA's tiles belong to a new chain almost every
// time, and each switch waited behind a CTA barrier for the new descriptor's
// round trip to L2).
template <class S, int V, bool WT, bool TOR = false>
__global__ void __launch_bounds__(TickBounds<V>::kThreads, TickBounds<V>::kMinBlocks) k_tick(EngineArgs ea) {
  constexpr bool MC = TOR && V == 0 && std::is_same<S, StoreF32x12>::value;
  __shared__ std::conditional_t<MC, ChainStaging, NoStaging> stg;
  __shared__ ChainDesc sd;
  __shared__ ChainState ss;  // the current chain's current state
  __shared__ int s_par;      // the state slot that holds the current states
  __shared__ double s_red[32];
  // Launched as a programmatic dependent (pdl), this tick may be scheduled
  // before the previous kernel of the stream has finished: wait for its
  // completion and memory before touching anything, then let the next tick
  // be scheduled.  Both are no-ops for an ordinary launch.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int total = ea.hdr->total_tiles;
  const int nchains = ea.hdr->nchains;
  int cur = -1;
  uint32_t np = 0, na = 0;  // FHKP counters of the current chain, flushed per warp
  bool wrote_partials = false;  // this thread wrote data that the last warp reads
  bool staged = false;  // (MC) stg holds the chain of this CTA's next tile
  for (int t = blockIdx.x; t < total; t += gridDim.x) {
    const int c = ea.tile_chain[t];  // the same for every thread of the CTA
    int cn = -1;  // (MC) the chain of the CTA's next tile
    if constexpr (MC) cn = t + (int)gridDim.x < total ? ea.tile_chain[t + gridDim.x] : -1;
    if (c != cur) {
      if (cur >= 0) flush_counters(sd, np, na);
      if constexpr (MC)
        if (staged) asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();  // every warp is done with the previous descriptor (MC: staged copies visible)
      if constexpr (MC) {
        if (staged)
          take_staged(sd, ss, stg);
        else
          load_chain(ea, c, sd, ss, s_par);
      } else {
        load_chain(ea, c, sd, ss, s_par);
      }
      __syncthreads();
      cur = c;
    }
    if constexpr (MC) {
      // the next tile belongs to another chain: stage it now (its buffer was
      // last read between the barriers above)
      staged = cn >= 0 && cn != c;
      if (staged) stage_chain(ea, cn, s_par, stg);
    }
    if (!ss.active) continue;
    const int lt = t - sd.tile_base;
    if (ss.stage < 2 * sd.D) {
      const int colour = ss.stage / sd.D, mu = ss.stage - colour * sd.D;
      update_tile<S, V, WT, false, TOR>(sd, ss.sweep, colour, mu, lt, np, na);
      continue;
    }
    const int layer = lt / sd.tiles_per_vl;
    const int tile = (int)blockDim.x / (V == kCoopVariant ? kCoopLanes : 1);
    const int jj = (lt - layer * sd.tiles_per_vl) * tile + threadIdx.x;
    const bool valid = (int)threadIdx.x < tile && jj < sd.Vn;
    if (ss.stage == kStageReunit) {
      if (valid) reunit_site<S>(sd, layer, jj);
    } else {
      double v[kPartVals] = {0, 0, 0, 0};
      if (valid) measure_site<S>(sd, layer, jj, v);
      block_reduce(v, s_red);
      if (threadIdx.x == 0 && in_bounds(lt, sd.nlayers * sd.tiles_per_layer, kBoundsPartial)) {
        for (int k = 0; k < kPartVals; ++k) sd.partials[(size_t)lt * kPartVals + k] = v[k];
        wrote_partials = true;
      }
    }
  }
  if (cur >= 0) flush_counters(sd, np, na);
  // The end of the launch's stage machine.  Counting warps, not CTAs, lets a
  // warp leave as soon as its own work is done (no CTA-wide barrier at the
  // end).  Writers of what a later warp of this launch reads (measurement
  // partials; with several chains also next states and the measuring list)
  // fence before counting (release); link stores and counter adds are
  // ordered for the next launch by the launch boundary.
  // One chain: the last warp to finish advances it in place, from its CTA's
  // shared copies (no global reads); the parity stays.  Every warp of a
  // one-chain launch takes this path, so that exactly one count per warp
  // is made.
  // Several chains: the first warp to finish writes every chain's next state
  // into the chain's other state slot (the current slot is only read during
  // a launch, so this overlaps the tiles still running) and lists the chains
  // that measure in this tick; then it counts itself a second time.  The
  // warp whose count completes the grid's warps + 1 finishes those
  // measurements and flips the parity.  (Reading and advancing hundreds of
  // chain states at the end of the launch, by the last warp, had kept the
  // rest of the GPU idle for several microseconds per tick.)
  const int lane = threadIdx.x & 31;
  const uint32_t nwarps = gridDim.x * (blockDim.x >> 5);
  constexpr uint32_t kMeasFlag = 0x80000000u;
  uint32_t prev = 0;
  if (lane == 0) {
    if (wrote_partials) __threadfence();
    prev = atomicAdd(&ea.hdr->done, 1u);
  }
  prev = __shfl_sync(0xffffffffu, prev, 0);
  const int par = cur >= 0 ? s_par : __ldcg(&ea.hdr->parity);
  if (nchains == 1) {
    if (prev != nwarps - 1) return;
    // (a CTA of a grid captured for more tiles than the engine now has can
    // have run no tile: it reads the chain from global memory)
    if (cur == 0)
      finish_single_chain(ea, sd, ss, par, lane);
    else
      finish_single_chain(ea, ea.desc[0], ea.state[par], par, lane);
    return;
  }
  int nmeas = -1;  // known to the first warp; the others read it when flagged
  if (prev == 0) {
    nmeas = 0;
    {
      // every chain's state read once, four per lane in flight; the
      // measuring chains listed in chain order (ballot prefix)
      constexpr int kU = 4;
      for (int base = 0; base < nchains; base += 32 * kU) {
        ChainState st[kU];
        StageParams sp[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          const int c = base + 32 * u + lane;
          if (c < nchains) {
            st[u] = ea.state[2 * (size_t)c + par];
            const ChainDesc &d = ea.desc[c];
            sp[u] = StageParams{d.D, d.reunit_every, d.measure_every};
          }
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          const int c = base + 32 * u + lane;
          const bool m = c < nchains && measures(st[u]);
          const unsigned mask = __ballot_sync(0xffffffffu, m);
          if (m) {
            const int slot = nmeas + __popc(mask & ((1u << lane) - 1u));
            if (in_bounds(slot, nchains, kBoundsSlot)) ea.meas_list[slot] = c;
          }
          nmeas += __popc(mask);
          if (c < nchains) ea.state[2 * (size_t)c + (par ^ 1)] = next_state(sp[u], st[u]);
        }
      }
    }
    if (lane == 0) ea.hdr->n_meas = nmeas;
    __threadfence();  // each lane's next states and list entries before the count
    __syncwarp();
    if (lane == 0) prev = atomicAdd(&ea.hdr->done, 1u | (nmeas ? kMeasFlag : 0u));
    prev = __shfl_sync(0xffffffffu, prev, 0);
  }
  if ((prev & ~kMeasFlag) != nwarps) return;
  // The last count: finish the listed measurements, flip the parity.
  if (nmeas < 0) nmeas = (prev & kMeasFlag) ? -2 : 0;
  if (nmeas != 0) {
    __threadfence();  // acquire the tiles' partials, the list and its length
    if (nmeas < 0) nmeas = __ldcg(&ea.hdr->n_meas);
    for (int i = 0; i < nmeas && i < nchains; ++i) {
      const int c = __ldcg(ea.meas_list + i);
      if (!in_bounds(c, nchains, kBoundsSlot)) continue;
      const ChainDesc &d = ea.desc[c];
      // the current slot: this tick's measurement count and anchor
      const ChainState &s = ea.state[2 * (size_t)c + par];
      double *out = d.results + (size_t)(s.n_meas % (uint32_t)d.result_cap) * (d.nlayers + 1) * kMeasVals;
      finalize_measure(d, d.partials, out);
      if (s.anchor) restart_bookkeeping(d, out);
    }
  }
  if (lane == 0) {
    ea.hdr->parity = par ^ 1;
    ea.hdr->done = 0u;
  }
}

// ------------------------------------------------------------------ launchers

// Tick kernel forms: FP32 12-real has variants 0..4 (TickBounds), FP32
// 18-real variant 0 only, FP64 one form (10; kMixedVariant with two-coupling
// chains) and, as the launcher's variant 1 (not a choice of the caller), eight
// lanes per link.
int tick_variants(int storage) { return storage == 1 ? 5 : 1; }

template <class S, int V, bool WT, bool TOR>
struct TickLaunch {
  static cudaError_t run(const EngineArgs *ea, int grid, int block, cudaStream_t st, bool pdl) {
    return launch_ex(k_tick<S, V, WT, TOR>, dim3((unsigned)grid), block, st, pdl, *ea);
  }
};
template <class S, int V, bool WT, bool TOR>
struct TickOccupancy {
  static cudaError_t run(int block, int *ctas) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, k_tick<S, V, WT, TOR>, block, 0);
  }
};

int tick_max_threads(int storage, int variant) {
  if (storage == 0) return TickBounds<10>::kThreads;
  if (variant == kFloatParked1) return kParkedThreads1;
  if (storage == 2 || variant >= kFloatLanes) return TickBounds<0>::kThreads;
  switch (variant) {
    case 0: return TickBounds<0>::kThreads;
    case 1: return TickBounds<1>::kThreads;
    case 2: return TickBounds<2>::kThreads;
    case 3: return TickBounds<3>::kThreads;
    default: return TickBounds<4>::kThreads;
  }
}

// One switch for launching and for occupancy queries: OP<S, V, WT, TOR>.  The
// torus form exists for the unrolled float variants (FP32 12-real 0 and 1,
// FP32 18-real 0); the others ignore `torus`.
template <template <class, int, bool, bool> class OP, bool WT, class... A>
static cudaError_t tick_dispatch(int storage, int variant, bool torus, A... a) {
  constexpr bool kT = !WT;  // a two-coupling chain is no torus
  const bool tor = torus && !WT;
  if (storage == 0) {
    if (variant == 1 && !WT) return OP<StoreF64x18, kCoopVariant, false, false>::run(a...);
    return OP<StoreF64x18, WT ? kMixedVariant : 10, WT, false>::run(a...);
  }
  if (storage == 2) return tor ? OP<StoreF32x18, 0, false, kT>::run(a...) : OP<StoreF32x18, 0, WT, false>::run(a...);
  switch (variant) {
    case 0: return tor ? OP<StoreF32x12, 0, false, kT>::run(a...) : OP<StoreF32x12, 0, WT, false>::run(a...);
    case 1: return tor ? OP<StoreF32x12, 1, false, kT>::run(a...) : OP<StoreF32x12, 1, WT, false>::run(a...);
    case 2: return OP<StoreF32x12, 2, WT, false>::run(a...);
    case 3: return OP<StoreF32x12, 3, WT, false>::run(a...);
    default: return OP<StoreF32x12, 4, WT, false>::run(a...);
  }
}

cudaError_t launch_tick(int storage, int variant, bool weighted, bool torus, const EngineArgs &ea, int grid, int block,
                        cudaStream_t st, bool pdl) {
  if (block > tick_max_threads(storage, variant)) return cudaErrorInvalidConfiguration;
  const EngineArgs *pa = &ea;
  return weighted ? tick_dispatch<TickLaunch, true>(storage, variant, torus, pa, grid, block, st, pdl)
                  : tick_dispatch<TickLaunch, false>(storage, variant, torus, pa, grid, block, st, pdl);
}

cudaError_t tick_occupancy(int storage, int variant, bool weighted, bool torus, int block, int *ctas_per_sm) {
  *ctas_per_sm = 0;
  if (block > tick_max_threads(storage, variant)) return cudaSuccess;
  return weighted ? tick_dispatch<TickOccupancy, true>(storage, variant, torus, block, ctas_per_sm)
                  : tick_dispatch<TickOccupancy, false>(storage, variant, torus, block, ctas_per_sm);
}

void host_advance_stage(const ChainDesc &d, ChainState &s) { advance_stage(d, s); }

cudaError_t bounds_record_tick(unsigned long long out[3]) {
  out[0] = out[1] = out[2] = 0;
#ifdef SU3_DEBUG_BOUNDS
  return cudaMemcpyFromSymbol(out, g_bounds, 3 * sizeof(unsigned long long));
#else
  return cudaSuccess;
#endif
}

}  // namespace su3g
