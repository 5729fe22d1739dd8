// su3_kernels.cu -- the kernels beside the chains' stages (sm_103a).
//
// k_start, k_convert, k_halo, k_sub_copy, k_measure_noalloc: start
//   configurations, canonical-layout conversion, the boxes of a divided
//   lattice and measurements of links the caller holds.
#include <cstdio>
#include <mutex>
#include <type_traits>

#include <cuda.h>  // CUcontext / CUresult for the two driver calls reached through the runtime

#include "su3_launch.h"
#include "su3_site.cuh"

namespace su3g {

// ------------------------------------------------------------------ one-off kernels

// Sum of a chain's booked action changes, one warp, fixed order.
__global__ void k_action_sum(const double *slots, int n, double *out) {
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += 32) v += slots[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (threadIdx.x == 0) *out = v;
}

// Arm every chain of an engine for n more sweeps, in stream order (the host
// mirror does the same): no host buffer, so nothing to synchronise on.
// Both state slots of a chain hold its current state between launches
// as far as the host-visible fields go: arm them both (the next launch
// overwrites the one that is not current).
__global__ void k_arm(ChainState *state, int nchains, uint32_t n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 2 * nchains; i += gridDim.x * blockDim.x) {
    ChainState s = state[i];
    s.target = s.sweep + n;
    s.active = 1;
    state[i] = s;
  }
}

// Set the bookkeeping-restart flag of one chain (both state slots), in
// stream order.
__global__ void k_set_anchor(ChainState *state, int value) {
  state[0].anchor = value;
  state[1].anchor = value;
}

cudaError_t launch_set_anchor(ChainState *state, int value, cudaStream_t st) {
  k_set_anchor<<<1, 1, 0, st>>>(state, value);
  return cudaGetLastError();
}

cudaError_t launch_arm(ChainState *state, int nchains, uint32_t n, cudaStream_t st) {
  if (nchains <= 0) return cudaSuccess;
  const int grid = (nchains + 255) / 256 < 1024 ? (nchains + 255) / 256 : 1024;
  k_arm<<<grid, 256, 0, st>>>(state, nchains, n);
  return cudaGetLastError();
}

cudaError_t launch_action_sum(const double *slots, int n, double *out, cudaStream_t st) {
  k_action_sum<<<1, 32, 0, st>>>(slots, n, out);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ start configurations

template <class S>
__global__ void k_start(const __grid_constant__ ChainDesc d, int hot) {
  const size_t nl = (size_t)d.nlayers * 2 * d.D * d.Vh;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nl; i += (size_t)gridDim.x * blockDim.x) {
    const int jj = (int)(i % d.Vh);
    size_t r = i / d.Vh;
    const int mu = (int)(r % d.D);
    r /= d.D;
    const int colour = (int)(r % 2);
    const int layer = (int)(r / 2);
    M3<double> m = m3_zero<double>();
    if (!hot) {
      m.e[0][0].re = m.e[1][1].re = m.e[2][2].re = 1.0;
    } else {
      // Haar SU(3): Gaussian rows 1, 2 (Box-Muller), Gram-Schmidt, cross product.
      const SiteGeo g = site_of(d, layer, colour, jj);
      const uint32_t key = site_key(d, g);
      double gs[12];
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const uint4 w = philox4x32_10(make_uint4(key, (uint32_t)mu, (uint32_t)b, kPurposeStart),
                                      make_uint2(d.seed_lo, d.seed_hi));
        const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          const double rad = sqrt(-2.0 * log(unif_d(ws[2 * p])));
          double sn, cs;
          sincospi(2.0 * unif_d(ws[2 * p + 1]), &sn, &cs);
          gs[4 * b + 2 * p] = rad * cs;
          gs[4 * b + 2 * p + 1] = rad * sn;
        }
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        m.e[0][k] = {gs[2 * k], gs[2 * k + 1]};
        m.e[1][k] = {gs[6 + 2 * k], gs[6 + 2 * k + 1]};
      }
      reunit_d(m);
    }
    S::store(plane_ptr<S>(d, layer, colour, mu), d.Vh, jj, m3_cast<typename S::R>(m));
  }
}

// ------------------------------------------------------------------ canonical layout <-> storage

template <class S>
__global__ void k_convert(const __grid_constant__ ChainDesc d, double *canon, int to_canonical) {
  const size_t nlinks = (size_t)d.nlayers * d.V * d.D;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nlinks; i += (size_t)gridDim.x * blockDim.x) {
    const int mu = (int)(i % d.D);
    const size_t ls = i / d.D;
    const int s = (int)(ls % d.V);
    const int layer = (int)(ls / d.V);
    // colour of site s: parity of its coordinate sum
    int r = s, sum = 0;
    for (int k = 0; k < d.D; ++k) {
      const int n = d.dims[k];
      sum += r % n;
      r /= n;
    }
    const int colour = sum & 1;
    typename S::Vec *p = plane_ptr<S>(d, layer, colour, mu);
    double *c = canon + i * 18;
    if (to_canonical) {
      const M3<typename S::R> m = S::load(p, d.Vh, s >> 1);
      for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) {
          c[(a * 3 + b) * 2] = (double)m.e[a][b].re;
          c[(a * 3 + b) * 2 + 1] = (double)m.e[a][b].im;
        }
    } else {
      M3<typename S::R> m;
      for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) m.e[a][b] = {(typename S::R)c[(a * 3 + b) * 2], (typename S::R)c[(a * 3 + b) * 2 + 1]};
      S::store(p, d.Vh, s >> 1, m);
    }
  }
}

// ------------------------------------------------------------------ sublattice boxes
// The paper's boundary exchange (Sec. 2.4: faces, and corners when two or
// more directions are divided) restated as device copies: every halo site
// of every box takes its links from the interior site that owns it in the
// undivided lattice (periodic wrap; a wrap across a glued boundary of the
// double-layered torus lands in the other layer).  Halo sites are never
// sources, so the copies do not race.

// Refresh every halo of a divided chain.  Threads run over the box's list of
// halo sites (blockIdx.y = box).
template <class S>
__global__ void k_halo(const __grid_constant__ ChainDesc d) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int count = d.halo_n[0] + d.halo_n[1];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < count; e += gridDim.x * blockDim.x)
    halo_copy<S>(d, blockIdx.y, e);
}

// Copy links between the undivided layout (plain) and the sublattice boxes
// (sub): to_sub = 1 scatters into the box interiors, 0 gathers from them.
template <class S>
__global__ void k_sub_copy(const ChainDesc *sub_dev, const ChainDesc *plain_dev, int to_sub) {
  const ChainDesc &d = *sub_dev;
  const ChainDesc &p = *plain_dev;
  const size_t nlinks = (size_t)p.nlayers * p.V * p.D;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nlinks; i += (size_t)gridDim.x * blockDim.x) {
    const int mu = (int)(i % p.D);
    const size_t ls = i / p.D;
    const int s = (int)(ls % p.V);
    const int L = (int)(ls / p.V);
    int r = s, par = 0, b = 0, bmul = 1, sp = 0;
    for (int k = 0; k < p.D; ++k) {
      const int gx = r % p.dims[k];
      r /= p.dims[k];
      par += gx;
      const int bo = gx / d.idims[k];
      b += bo * bmul;
      bmul *= d.bdiv[k];
      sp += (gx - bo * d.idims[k] + d.hpad[k]) * d.stride[k];
    }
    const int colour = par & 1;
    typename S::Vec *pv = plane_ptr<S>(p, L, colour, mu);
    typename S::Vec *sv = plane_ptr<S>(d, L * d.nb + b, colour, mu);
    if (to_sub)
      S::copy(sv, d.Vh, sp >> 1, pv, p.Vh, s >> 1);
    else
      S::copy(pv, p.Vh, s >> 1, sv, d.Vh, sp >> 1);
  }
}

// Links given as rows 1 and 2 in float (12 per link, canonical site order:
// [layer][i_s - 1][mu][row][col][re, im]); row 3 = conj(row1 x row2).
template <class S>
__global__ void k_convert_rows2(const __grid_constant__ ChainDesc d, const float *src) {
  const size_t nlinks = (size_t)d.nlayers * d.V * d.D;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nlinks; i += (size_t)gridDim.x * blockDim.x) {
    const int mu = (int)(i % d.D);
    const size_t ls = i / d.D;
    const int s = (int)(ls % d.V);
    const int layer = (int)(ls / d.V);
    int r = s, sum = 0;
    for (int k = 0; k < d.D; ++k) {
      const int n = d.dims[k];
      sum += r % n;
      r /= n;
    }
    const float4 *c = reinterpret_cast<const float4 *>(src + i * 12);
    const float4 q0 = c[0], q1 = c[1], q2 = c[2];
    using R = typename S::R;
    M3<R> m;
    m.e[0][0] = {(R)q0.x, (R)q0.y};
    m.e[0][1] = {(R)q0.z, (R)q0.w};
    m.e[0][2] = {(R)q1.x, (R)q1.y};
    m.e[1][0] = {(R)q1.z, (R)q1.w};
    m.e[1][1] = {(R)q2.x, (R)q2.y};
    m.e[1][2] = {(R)q2.z, (R)q2.w};
    third_row(m);
    S::store(plane_ptr<S>(d, layer, sum & 1, mu), d.Vh, s >> 1, m);
  }
}

// ------------------------------------------------------------------ measurement without allocation
// For callers that cannot allocate device memory (see su3_measure_noalloc):
// the per-tile partial sums go to a fixed array in the library's own device
// memory instead of a buffer from cudaMalloc.  Every tile writes its own
// slots before the finishing kernel reads them, so nothing has to start at
// zero; calls that overlap on the GPU share the array and race.

constexpr int kNoAllocTiles = 32768;  // 32768 tiles x 4 doubles = 1 MiB
static __device__ __align__(256) double g_noalloc_partials[kNoAllocTiles * kPartVals];

template <class S>
__global__ void __launch_bounds__(256) k_measure_noalloc(ChainDesc d, double *partials) {
  __shared__ double s_red[32];
  const int total = d.tiles_per_layer * d.nlayers;
  for (int lt = blockIdx.x; lt < total; lt += gridDim.x) {
    const int layer = lt / d.tiles_per_layer;
    const int jj = (lt - layer * d.tiles_per_layer) * blockDim.x + threadIdx.x;
    double v[kPartVals] = {0, 0, 0, 0};
    if (jj < d.Vh) measure_site<S>(d, layer, jj, v);
    block_reduce(v, s_red);
    if (threadIdx.x == 0 && in_bounds(lt, kNoAllocTiles, kBoundsPartial))
      for (int k = 0; k < kPartVals; ++k) partials[(size_t)lt * kPartVals + k] = v[k];
  }
}

__global__ void k_measure_finalize_noalloc(ChainDesc d, const double *partials, double *out) {
  finalize_measure(d, partials, out);
}

int noalloc_max_tiles() { return kNoAllocTiles; }

// The unique id of the current context (cuCtxGetId), or 0 when there is no
// current context or the driver cannot say.  The two driver calls are
// reached through the runtime's entry-point table, so the library does not
// link the driver library itself.
static unsigned long long current_context_id() {
  using GetCurrent = CUresult (*)(CUcontext *);
  using GetId = CUresult (*)(CUcontext, unsigned long long *);
  static GetCurrent get_current = nullptr;
  static GetId get_id = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_current = reinterpret_cast<GetCurrent>(p);
    p = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_id = reinterpret_cast<GetId>(p);
  });
  CUcontext ctx = nullptr;
  unsigned long long id = 0;
  if (!get_current || !get_id || get_current(&ctx) != CUDA_SUCCESS || !ctx || get_id(ctx, &id) != CUDA_SUCCESS)
    return 0;
  return id;
}

// Device address of the scratch array in the current context.  Host code
// cannot use the symbol itself (it names a host-side stand-in), so the
// address is looked up with cudaGetSymbolAddress.  It is kept per device
// together with the id of the context it was taken in: a device reset
// (cudaDeviceReset) or any other teardown of the context unloads the
// library's module, and the next call then sees a new context id and looks
// the address up again instead of using a stale one.  Without a context id
// the address is looked up on every call.
static cudaError_t noalloc_scratch(double **ptr) {
  static std::mutex mu;
  static double *addr[64] = {nullptr};
  static unsigned long long ctx_of[64] = {0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(mu);
  const unsigned long long id = current_context_id();
  if (id && ctx_of[dev] == id && addr[dev]) {
    *ptr = addr[dev];
    return cudaSuccess;
  }
  void *p = nullptr;
  e = cudaGetSymbolAddress(&p, g_noalloc_partials);  // also makes the device's context current
  if (e != cudaSuccess) return e;
  addr[dev] = static_cast<double *>(p);
  ctx_of[dev] = current_context_id();
  *ptr = addr[dev];
  return cudaSuccess;
}

cudaError_t launch_measure_noalloc(int storage, const ChainDesc &d, int block, double *out, cudaStream_t st) {
  double *partials = nullptr;
  cudaError_t e = noalloc_scratch(&partials);
  if (e != cudaSuccess) return e;
  const int tiles = d.tiles_per_layer * d.nlayers;
  const int grid = tiles < 4096 ? tiles : 4096;
  return by_storage(storage, [&](auto s) {
    k_measure_noalloc<decltype(s)><<<grid, block, 0, st>>>(d, partials);
    k_measure_finalize_noalloc<<<1, 32, 0, st>>>(d, partials, out);
    return cudaGetLastError();
  });
}

// ------------------------------------------------------------------ debug bounds checks (host side)

// A deliberate out-of-range index checked by the device predicate; nothing
// is accessed, only the violation record is written.
__global__ void k_bounds_selftest() { (void)in_bounds(1, 1, kBoundsSelfTest); }

bool debug_bounds_build() {
#ifdef SU3_DEBUG_BOUNDS
  return true;
#else
  return false;
#endif
}

cudaError_t bounds_record(unsigned long long out[3]) {
  out[0] = out[1] = out[2] = 0;
#ifdef SU3_DEBUG_BOUNDS
  return cudaMemcpyFromSymbol(out, g_bounds, 3 * sizeof(unsigned long long));
#else
  return cudaSuccess;
#endif
}

cudaError_t launch_bounds_selftest() {
  k_bounds_selftest<<<1, 1>>>();
  cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : cudaDeviceSynchronize();
}

// ------------------------------------------------------------------ launchers

cudaError_t launch_halo(int storage, const ChainDesc &d, int halo_sites, cudaStream_t st, bool pdl) {
  const int block = 256;
  const dim3 grid((unsigned)((halo_sites + block - 1) / block > 0 ? (halo_sites + block - 1) / block : 1),
                  (unsigned)(d.nlayers * d.nb));
  return by_storage(storage, [&](auto s) { return launch_ex(k_halo<decltype(s)>, grid, block, st, pdl, d); });
}

static int copy_grid(size_t nlinks, int block) {
  return (int)((nlinks + block - 1) / block < 65536 ? (nlinks + block - 1) / block : 65536);
}

cudaError_t launch_sub_copy(int storage, const ChainDesc *sub_dev, const ChainDesc *plain_dev, size_t nlinks,
                            int to_sub, cudaStream_t st) {
  const int block = 256, grid = copy_grid(nlinks, block);
  return by_storage(storage, [&](auto s) {
    k_sub_copy<decltype(s)><<<grid, block, 0, st>>>(sub_dev, plain_dev, to_sub);
    return cudaGetLastError();
  });
}

cudaError_t launch_start(int storage, const ChainDesc &d, size_t nlinks, int hot, cudaStream_t st) {
  const int block = 256, grid = copy_grid(nlinks, block);
  return by_storage(storage, [&](auto s) {
    k_start<decltype(s)><<<grid, block, 0, st>>>(d, hot);
    return cudaGetLastError();
  });
}

cudaError_t launch_convert_rows2(int storage, const ChainDesc &d, size_t nlinks, const float *src, cudaStream_t st) {
  const int block = 256, grid = copy_grid(nlinks, block);
  return by_storage(storage, [&](auto s) {
    k_convert_rows2<decltype(s)><<<grid, block, 0, st>>>(d, src);
    return cudaGetLastError();
  });
}

cudaError_t launch_convert(int storage, const ChainDesc &d, size_t nlinks, double *canon, int to_canonical,
                           cudaStream_t st) {
  const int block = 256, grid = copy_grid(nlinks, block);
  return by_storage(storage, [&](auto s) {
    k_convert<decltype(s)><<<grid, block, 0, st>>>(d, canon, to_canonical);
    return cudaGetLastError();
  });
}

}  // namespace su3g
