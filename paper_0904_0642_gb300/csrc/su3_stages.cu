// su3_stages.cu -- the re-unitarisation and the measurement of one chain
// (sm_103a).
#include "su3_launch.h"
#include "su3_site.cuh"

namespace su3g {

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

cudaError_t bounds_record_stages(unsigned long long out[3]) {
  out[0] = out[1] = out[2] = 0;
#ifdef SU3_DEBUG_BOUNDS
  return cudaMemcpyFromSymbol(out, g_bounds, 3 * sizeof(unsigned long long));
#else
  return cudaSuccess;
#endif
}

}  // namespace su3g
