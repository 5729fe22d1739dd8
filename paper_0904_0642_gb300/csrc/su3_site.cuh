// su3_site.cuh -- device code of one site: geometry and neighbours, the link
// update in its forms, re-unitarisation and measurement.  Included by the
// kernels of one chain (su3_phase.cuh) and of many (su3_tick.cu).
#pragma once
#include <type_traits>
#include <utility>

#include "su3_device.cuh"
#include "su3_fixed.cuh"

namespace su3g {

// ------------------------------------------------------------------ geometry

struct SiteGeo {
  int x[kMaxD];
  int s;      // i_s - 1 within the layer
  int layer;
};

__device__ __forceinline__ int fast_div(int r, const FastDiv &f) {
  return (int)((__umulhi(f.m, (uint32_t)r) + (uint32_t)r) >> f.s);
}

// Coordinates of the site of colour `colour` at checkerboard index jj
// (eqs. xD, x^i, i_c): the even lexicographic index 2 jj shares its row
// with the odd one, and the colour fixes which of the two it is.
// SUB (sublattice boxes): jj counts the interior sites of the box; the
// returned coordinates and index are those of the padded box.  Sublattice
// origins are even, so the colour is the colour of the undivided lattice.
template <bool SUB = false>
__device__ __forceinline__ SiteGeo site_of(const ChainDesc &d, int layer, int colour, int jj) {
  SiteGeo g;
  if constexpr (SUB) {
    int r = 2 * jj, par = colour;
#pragma unroll
    for (int i = 0; i < kMaxD; ++i) {
      if (i < d.D) {
        const int n = d.idims[i];
        const int q = fast_div(r, d.idiv[i]);
        g.x[i] = r - q * n;
        r = q;
        if (i > 0) par += g.x[i];
      } else {
        g.x[i] = 0;
      }
    }
    g.x[0] += par & 1;
    int sp = 0;
#pragma unroll
    for (int i = 0; i < kMaxD; ++i)
      if (i < d.D) {
        g.x[i] += d.hpad[i];
        sp += g.x[i] * d.stride[i];
      }
    g.s = sp;
    g.layer = layer;
    return g;
  }
  int r = 2 * jj;
  int par = colour;
  if (d.pow2) {
#pragma unroll
    for (int i = 0; i < kMaxD; ++i) {
      if (i < d.D) {
        g.x[i] = r & (d.dims[i] - 1);
        r >>= d.shift[i];
        if (i > 0) par += g.x[i];
      } else {
        g.x[i] = 0;
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < kMaxD; ++i) {
      if (i < d.D) {
        const int n = d.dims[i];
        const int q = fast_div(r, d.idiv[i]);
        g.x[i] = r - q * n;
        r = q;
        if (i > 0) par += g.x[i];
      } else {
        g.x[i] = 0;
      }
    }
  }
  par &= 1;
  g.x[0] += par;
  g.s = 2 * jj + par;
  g.layer = layer;
  return g;
}

// Lexicographic offset and layer flip of one step in direction nu.
__device__ __forceinline__ void step_fwd(const ChainDesc &d, int xnu, int nu, int &off, int &flip) {
  const int n = d.dims[nu], st = d.stride[nu];
  if (xnu == n - 1) {
    off = -(n - 1) * st;
    flip = (d.nlayers == 2) ? ((d.glue_mask >> nu) & 1) : 0;
  } else {
    off = st;
    flip = 0;
  }
}
__device__ __forceinline__ void step_bwd(const ChainDesc &d, int xnu, int nu, int &off, int &flip) {
  const int n = d.dims[nu], st = d.stride[nu];
  if (xnu == 0) {
    off = (n - 1) * st;
    flip = (d.nlayers == 2) ? ((d.glue_mask >> nu) & 1) : 0;
  } else {
    off = -st;
    flip = 0;
  }
}

// The layer reached by a step with layer flip f: for sublattice boxes the
// virtual layer of the same sublattice in the other layer.
template <bool SUB>
__device__ __forceinline__ int lflip(const ChainDesc &d, int l, int f) {
  if constexpr (SUB)
    return f ? (l < d.nb ? l + d.nb : l - d.nb) : l;
  else
    return l ^ f;
}

// 1 when (virtual) layer l belongs to layer 1 of the double-layered torus.
template <bool SUB>
__device__ __forceinline__ int in_layer1(const ChainDesc &d, int l) {
  if constexpr (SUB)
    return l >= d.nb ? 1 : 0;
  else
    return l;
}

// The places where a site's links are stored: f(box, checkerboard index) for
// the site itself (m = 0) and, SUB, for its copies in the halos of the
// neighbouring boxes (one per nonempty set m of divided directions in which
// it lies on a face).  m runs from `first` in steps of `step`, so that lanes
// can share the stores.  An update phase writes the copies of its own links
// itself: no link of the phase's colour and direction is read in it.  A site
// on the high (low) face of direction k appears in the low (high) halo of the
// next (previous) box; a step across a glued boundary of the double-layered
// torus lands in the other layer.
template <bool SUB, class F>
__device__ __forceinline__ void for_replicas(const ChainDesc &d, const SiteGeo &g, int first, int step, F &&f) {
  if constexpr (!SUB) {
    if (first == 0) f(g.layer, g.s >> 1);
  } else {
    int on = 0;  // directions in which the site lies on a face
#pragma unroll
    for (int k = 0; k < kMaxD; ++k)
      if (k < d.D && d.hpad[k] && (g.x[k] == 1 || g.x[k] == d.idims[k])) on |= 1 << k;
    const int L = g.layer / d.nb, b = g.layer - L * d.nb;
#pragma unroll 1
    for (int m = first; m < (1 << kMaxD); m += step) {
      if (m & ~on) continue;
      int s = g.s, flip = 0, box = 0, mul = 1, rest = b;
#pragma unroll
      for (int k = 0; k < kMaxD; ++k)
        if (k < d.D) {
          const int rq = fast_div(rest, d.bdivf[k]);
          int bc = rest - rq * d.bdiv[k];
          rest = rq;
          if ((m >> k) & 1) {
            const bool low = g.x[k] == 1;
            s += (low ? d.idims[k] : -d.idims[k]) * d.stride[k];  // 1 -> n + 1, n -> 0
            bc += low ? -1 : 1;
            if (bc < 0 || bc >= d.bdiv[k]) {
              bc = bc < 0 ? d.bdiv[k] - 1 : 0;
              if (d.nlayers == 2) flip ^= (d.glue_mask >> k) & 1;
            }
          }
          box += bc * mul;
          mul *= d.bdiv[k];
        }
      f((L ^ flip) * d.nb + box, s >> 1);
    }
  }
}

// Random-number site key: layer * V + i_s - 1, or the site number of
// (x mod period) on the period lattice (identical numbers on sublattices).
// SUB: from the coordinates in the undivided lattice, so that a divided
// lattice draws the same numbers as the undivided one.
template <bool SUB = false>
__device__ __forceinline__ uint32_t site_key(const ChainDesc &d, const SiteGeo &g) {
  if constexpr (SUB) {
    const int L = g.layer / d.nb;
    int b = g.layer - L * d.nb;
    const int lay = (d.nlayers == 2 && !d.layer_blind) ? L : 0;
    int key = 0;
#pragma unroll
    for (int i = 0; i < kMaxD; ++i)
      if (i < d.D) {
        const int q = fast_div(b, d.bdivf[i]), bc = b - q * d.bdiv[i];
        b = q;
        const int gx = bc * d.idims[i] + g.x[i] - d.hpad[i];
        key += d.custom_period ? (gx % d.period[i]) * d.pstride[i] : gx * d.gstride[i];
      }
    return (uint32_t)(lay * (d.custom_period ? d.Vp : d.V) + key);
  }
  const int lay = (d.nlayers == 2 && !d.layer_blind) ? g.layer : 0;
  if (!d.custom_period) return (uint32_t)(lay * d.V + g.s);
  int key = 0;
#pragma unroll
  for (int i = 0; i < kMaxD; ++i)
    if (i < d.D) key += (g.x[i] % d.period[i]) * d.pstride[i];
  return (uint32_t)(lay * d.Vp + key);
}

__device__ __forceinline__ int sel(const int (&x)[kMaxD], int i) {
  int v = 0;
#pragma unroll
  for (int k = 0; k < kMaxD; ++k)
    if (k == i) v = x[k];
  return v;
}

// ------------------------------------------------------------------ one link update

// The staples of one direction nu added to A.
template <class S, bool WT, bool SUB>
__device__ __forceinline__ void add_staples(const ChainDesc &d, const SiteGeo &g, int colour, int mu, int nu, int xnu,
                                            int sp, int lp, M3<typename S::R> &A) {
  using R = typename S::R;
  const int Vh = d.Vh, layer = g.layer, jj = g.s >> 1, oc = colour ^ 1;
  int offn, fln, offm, flm;
  step_fwd(d, xnu, nu, offn, fln);
  step_bwd(d, xnu, nu, offm, flm);
  const int sn = g.s + offn, ln = lflip<SUB>(d, layer, fln);  // x + nu
  const int sm = g.s + offm, lm = lflip<SUB>(d, layer, flm);  // x - nu
  const int spm = sp + offm, lpm = lflip<SUB>(d, lp, flm);    // x + mu - nu
  // upper staple U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+ = a (c b)^+, all factors SU(3):
  // two rows of each product, the third from the cross product
  const M3<R> b = S::load(plane_ptr<S>(d, ln, oc, mu), Vh, sn >> 1);       // U_mu(x+nu)
  const M3<R> c = S::load2(plane_ptr<S>(d, layer, colour, nu), Vh, jj);    // U_nu(x)
  M3<R> cb = mul_nn_2(c, b);
  third_row(cb);
  const M3<R> a = S::load2(plane_ptr<S>(d, lp, oc, nu), Vh, sp >> 1);      // U_nu(x+mu)
  // WT (a kernel compiled for two-coupling chains) and a two-coupling chain:
  // each staple enters with the coupling of its plaquette, beta1 when any of
  // its links lies in layer 1, so A carries the betas and the heatbath runs
  // with beta = 1.  Otherwise plain sums (beta enters the heatbath).
  const bool weighted = WT && d.weighted;
  const R b0 = sizeof(R) == 4 ? (R)d.beta_f : (R)d.beta_d, b1 = sizeof(R) == 4 ? (R)d.beta1_f : (R)d.beta1_d;
  if (weighted)
    acc_su3_2rows_w(A, mul_nd_2(a, cb), (in_layer1<SUB>(d, layer) | in_layer1<SUB>(d, lp) | in_layer1<SUB>(d, ln)) ? b1 : b0);
  else
    acc_su3_2rows(A, mul_nd_2(a, cb));
  // lower staple U_nu(x+mu-nu)^+ U_mu(x-nu)^+ U_nu(x-nu) = (e f)^+ h
  const M3<R> f = S::load(plane_ptr<S>(d, lpm, colour, nu), Vh, spm >> 1); // U_nu(x+mu-nu)
  const M3<R> e = S::load2(plane_ptr<S>(d, lm, oc, mu), Vh, sm >> 1);      // U_mu(x-nu)
  M3<R> ef = mul_nn_2(e, f);
  third_row(ef);
  const M3<R> h = S::load(plane_ptr<S>(d, lm, oc, nu), Vh, sm >> 1);       // U_nu(x-nu)
  if (weighted)
    acc_su3_2rows_w(A, mul_dn_2(ef, h), (in_layer1<SUB>(d, lm) | in_layer1<SUB>(d, lpm) | in_layer1<SUB>(d, layer)) ? b1 : b0);
  else
    acc_su3_2rows(A, mul_dn_2(ef, h));
}

// The staples of one direction nu from precomputed plane offsets (p*, in
// vectors from the chain's link base) and checkerboard indices (j*) of the
// six links: the arithmetic and its order are those of add_staples.  Plane
// offset and index stay separate because the 18-real float form addresses a
// plane's 16-byte vectors from its (16-byte aligned) start.
// Where a form's vectors are its addressing unit (every form but the 18-real
// float one) offset and index are summed first: one index per link.
template <class S>
__device__ __forceinline__ M3<typename S::R> load_at(const ChainDesc &d, const typename S::Vec *base, int Vh, int p,
                                                     int j, bool rows2) {
  // the plane offset lies within the (virtual) layers' planes
  if (!in_bounds(p, (long long)d.nlayers * d.nb * 2 * d.D * S::NQ * Vh, kBoundsLink)) return m3_zero<typename S::R>();
  if constexpr (sizeof(typename S::Vec) == 8)  // the 18-real float forms
    return rows2 ? S::load2(base + p, Vh, j) : S::load(base + p, Vh, j);
  else
  {
    if (!in_bounds(j, Vh, kBoundsIndex)) return m3_zero<typename S::R>();
    return rows2 ? S::load2(base + (p + j), Vh, 0) : S::load(base + (p + j), Vh, 0);
  }
}

template <class S, bool WT>
__device__ __forceinline__ void add_staples_idx(const ChainDesc &d, const typename S::Vec *base, int Vh, int pb, int jb,
                                                int pc, int jc, int pa, int ja, int pf, int jf, int pe, int je, int ph,
                                                int jh, int wu, int wl, M3<typename S::R> &A) {
  using R = typename S::R;
  const M3<R> b = load_at<S>(d, base, Vh, pb, jb, false);  // U_mu(x+nu)
  const M3<R> c = load_at<S>(d, base, Vh, pc, jc, true);   // U_nu(x)
  M3<R> cb = mul_nn_2(c, b);
  third_row(cb);
  const M3<R> a = load_at<S>(d, base, Vh, pa, ja, true);   // U_nu(x+mu)
  const bool weighted = WT && d.weighted;
  const R b0 = sizeof(R) == 4 ? (R)d.beta_f : (R)d.beta_d, b1 = sizeof(R) == 4 ? (R)d.beta1_f : (R)d.beta1_d;
  if (weighted)
    acc_su3_2rows_w(A, mul_nd_2(a, cb), wu ? b1 : b0);
  else
    acc_su3_2rows(A, mul_nd_2(a, cb));
  const M3<R> f = load_at<S>(d, base, Vh, pf, jf, false);  // U_nu(x+mu-nu)
  const M3<R> e = load_at<S>(d, base, Vh, pe, je, true);   // U_mu(x-nu)
  M3<R> ef = mul_nn_2(e, f);
  third_row(ef);
  const M3<R> h = load_at<S>(d, base, Vh, ph, jh, false);  // U_nu(x-nu)
  if (weighted)
    acc_su3_2rows_w(A, mul_dn_2(ef, h), wl ? b1 : b0);
  else
    acc_su3_2rows(A, mul_dn_2(ef, h));
}

// A thread's draws parked in shared memory, in slots of its own (no barrier).
constexpr int kParkedBytes = 9 * sizeof(float2);  // per thread
__device__ __forceinline__ float2 *parked_draws() {
  extern __shared__ float2 s_parked[];
  return s_parked + threadIdx.x;
}
__device__ __forceinline__ void park_draws(const DrawPre (&pre)[3]) {
  float2 *p = parked_draws();
#pragma unroll
  for (int g = 0; g < 3; ++g) {
    p[(3 * g) * blockDim.x] = make_float2(pre[g].L, pre[g].u4sq);
    p[(3 * g + 1) * blockDim.x] = make_float2(pre[g].costh, pre[g].sinth);
    p[(3 * g + 2) * blockDim.x] = make_float2(pre[g].cphi, pre[g].sphi);
  }
}
__device__ __forceinline__ void unpark_draws(DrawPre (&pre)[3]) {
  const float2 *p = parked_draws();
#pragma unroll
  for (int g = 0; g < 3; ++g) {
    const float2 a = p[(3 * g) * blockDim.x], b = p[(3 * g + 1) * blockDim.x], c = p[(3 * g + 2) * blockDim.x];
    pre[g] = DrawPre{a.x, a.y, b.x, b.y, c.x, c.y};
  }
}
struct NotEarly {
  __device__ __forceinline__ void operator()(int) const {}
};

// update_site for an undivided lattice with the neighbour geometry computed
// once per site: forward and backward site offsets and layer flips in every
// direction, and the plane offsets as multiples of one plane stride.  Same
// arithmetic, same order as update_site.
// EARLY 1: the draws first, in registers, and ready(nu) before the staples of
// a direction.  EARLY 2: the draws first, parked in shared memory (a thread's
// own slots) until the staples are summed, and ready(-1) before the staples.
template <class S, bool WT, int DF = 0, int EARLY = 0, class Ready = NotEarly>
__device__ __forceinline__ void update_site_lean(const ChainDesc &d, uint32_t sweep, int colour, int mu, int layer,
                                                 int jj, uint32_t &nprop, uint32_t &nacc, typename S::R &dretr,
                                                 Ready &&ready = Ready()) {
  using R = typename S::R;
  using Vec = typename S::Vec;
  // DF > 0: every chain of the launch is a periodic torus (one layer) of
  // dimension DF, undivided, with one coupling and the default random-number
  // site key (no layer flips, no layer offsets, D known to the compiler)
  constexpr bool kTorus = DF > 0;
  if constexpr (kTorus) layer = 0;
  const int Vh = d.Vh, D = kTorus ? DF : d.D;
  const SiteGeo g = site_of<false>(d, layer, colour, jj);
  const int PS = S::NQ * Vh, CS = D * PS, LS = 2 * CS;
  const int oc = colour ^ 1;
  const Vec *base = reinterpret_cast<const Vec *>(d.links);
  const int s = g.s;
  int of[kMaxD], ob[kMaxD], ff[kMaxD], fb[kMaxD];
#pragma unroll
  for (int k = 0; k < kMaxD; ++k) {
    of[k] = ob[k] = ff[k] = fb[k] = 0;
    if (k < D) {
      step_fwd(d, g.x[k], k, of[k], ff[k]);
      step_bwd(d, g.x[k], k, ob[k], fb[k]);
      if constexpr (kTorus) ff[k] = fb[k] = 0;
    }
  }
  int ofm = 0, ffm = 0;
#pragma unroll
  for (int k = 0; k < kMaxD; ++k)
    if (k == mu) {
      ofm = of[k];
      ffm = ff[k];
    }
  const int lp = layer ^ ffm;            // layer of x + mu
  const int sp = s + ofm;                // x + mu
  const int pmu_oc = oc * CS + mu * PS;  // plane (oc, mu) within a layer
  const uint2 key = make_uint2(d.seed_lo, d.seed_hi);
  const uint32_t skey = kTorus ? (uint32_t)s : site_key<false>(d, g);  // the torus form has the default key
  [[maybe_unused]] DrawPre pre[3];
  if constexpr (EARLY > 0) cm_draws_f(pre, key, skey, sweep, colour, mu);
  if constexpr (EARLY == 2) {
    park_draws(pre);
    ready(-1);
  }
  M3<R> A = m3_zero<R>();
#pragma unroll
  for (int nu = 0; nu < kMaxD; ++nu) {
    if (nu < D && nu != mu) {
      if constexpr (EARLY == 1) ready(nu);
      const int lb = layer ^ ff[nu], lm = layer ^ fb[nu], lf = lp ^ fb[nu];
      const int sm = s + ob[nu];
      add_staples_idx<S, WT>(d, base, Vh,
                             lb * LS + pmu_oc, (s + of[nu]) >> 1,                   // U_mu(x+nu)
                             layer * LS + colour * CS + nu * PS, jj,                // U_nu(x)
                             lp * LS + oc * CS + nu * PS, sp >> 1,                  // U_nu(x+mu)
                             lf * LS + colour * CS + nu * PS, (sp + ob[nu]) >> 1,   // U_nu(x+mu-nu)
                             lm * LS + pmu_oc, sm >> 1,                             // U_mu(x-nu)
                             lm * LS + oc * CS + nu * PS, sm >> 1,                  // U_nu(x-nu)
                             layer | lp | lb, lm | lf | layer, A);
    }
  }
  typename S::Vec *pu = plane_ptr<S>(d, layer, colour, mu);
  M3<R> U = S::load(pu, Vh, jj);
  const R beta = (WT && d.weighted) ? R(1) : (sizeof(R) == 4 ? (R)d.beta_f : (R)d.beta_d);
  if constexpr (EARLY == 2) unpark_draws(pre);
  if constexpr (EARLY > 0)
    cm_apply_f(U, A, beta, d.hits, key, skey, sweep, colour, mu, pre, nprop, nacc, dretr);
  else if constexpr (sizeof(R) == 4)
    cm_update_f(U, A, beta, d.hits, key, skey, sweep, colour, mu, nprop, nacc, dretr);
  else
    cm_update(U, A, beta, d.hits, key, skey, sweep, colour, mu, nprop, nacc, dretr);
  S::store(pu, Vh, jj, U);
}

// ROLLED: the loop over staple directions stays a loop (no unrolling), so the
// compiler cannot hoist later directions' loads; fewer registers, less code.
template <class S, bool ROLLED, bool WT, bool SUB, bool EARLY = false, class Ready = NotEarly>
__device__ __forceinline__ void update_site(const ChainDesc &d, uint32_t sweep, int colour, int mu, int layer, int jj,
                                            uint32_t &nprop, uint32_t &nacc, typename S::R &dretr,
                                            Ready &&ready = Ready()) {
  using R = typename S::R;
  const int Vh = d.Vh;
  const SiteGeo g = site_of<SUB>(d, layer, colour, jj);
  int offp, flp;
  step_fwd(d, sel(g.x, mu), mu, offp, flp);
  const int sp = g.s + offp, lp = lflip<SUB>(d, layer, flp);  // x + mu
  const uint2 key = make_uint2(d.seed_lo, d.seed_hi);
  const uint32_t skey = site_key<SUB>(d, g);

  [[maybe_unused]] DrawPre pre[3];
  if constexpr (EARLY) cm_draws_f(pre, key, skey, sweep, colour, mu);
  M3<R> A = m3_zero<R>();
  if constexpr (ROLLED) {
#pragma unroll 1
    for (int nu = 0; nu < d.D; ++nu)
      if (nu != mu) {
        ready(nu);
        add_staples<S, WT, SUB>(d, g, colour, mu, nu, sel(g.x, nu), sp, lp, A);
      }
  } else {
#pragma unroll
    for (int nu = 0; nu < kMaxD; ++nu)
      if (nu < d.D && nu != mu) add_staples<S, WT, SUB>(d, g, colour, mu, nu, g.x[nu], sp, lp, A);
  }
  typename S::Vec *pu = plane_ptr<S>(d, layer, colour, mu);
  const int ju = g.s >> 1;  // jj itself unless the site sits in a padded box
  M3<R> U = S::load(pu, Vh, ju);
  const R beta = (WT && d.weighted) ? R(1) : (sizeof(R) == 4 ? (R)d.beta_f : (R)d.beta_d);
  if constexpr (EARLY)
    cm_apply_f(U, A, beta, d.hits, key, skey, sweep, colour, mu, pre, nprop, nacc, dretr);
  else if constexpr (sizeof(R) == 4)
    cm_update_f(U, A, beta, d.hits, key, skey, sweep, colour, mu, nprop, nacc, dretr);
  else
    cm_update(U, A, beta, d.hits, key, skey, sweep, colour, mu, nprop, nacc, dretr);
  for_replicas<SUB>(d, g, 0, 1, [&](int vl, int j) { S::store(plane_ptr<S>(d, vl, colour, mu), Vh, j, U); });
}


// ------------------------------------------------------------------ float link update, eight lanes per link
// For lattices whose updates are bound by one thread's chain of ~2900
// dependent instructions.  Lane l forms the l-th staple product (rows 0, 1);
// the draws' counter-only parts of the three subgroups take one pass over the
// lanes; then every lane sums the staples in the order of update_site and
// runs the subgroups.  Same operations in the same order per element: the
// links are bitwise those of the other forms.  Called by whole warps; lanes
// without a link (valid false) run along on a repeated one.

// Lane l's part of the draws (no link is read): lanes 0..2 the first
// proposals, lanes 3, 4 the direction blocks; then lanes 3..5 the directions.
__device__ __forceinline__ DrawPre lanes_draws_f(uint2 key, uint32_t c0, uint32_t sweep, int colour, int mu) {
  const int lane = threadIdx.x & 31, l8 = lane & 7, base = lane & 24;
  const int sub = l8 < 3 ? l8 : (l8 < 6 ? l8 - 3 : 0);
  const uint32_t btag = heatbath_tag(colour, mu, l8 < 3 ? l8 : (l8 == 4 ? 2 : 0)) | (l8 < 3 ? 0u : kHitDirection);
  const uint4 w = philox4x32_10(make_uint4(c0, sweep, btag, kPurposeHeatbath), key);
  const int dl = base + (sub == 2 ? 4 : 3);
  const uint32_t d0 = __shfl_sync(0xffffffffu, w.x, dl), d1 = __shfl_sync(0xffffffffu, w.y, dl);
  const uint32_t d2 = __shfl_sync(0xffffffffu, w.z, dl), d3 = __shfl_sync(0xffffffffu, w.w, dl);
  DrawPre mine;
  proposal_pre_words(mine, w);
  direction_pre_f(mine, sub == 1 ? d2 : d0, sub == 1 ? d3 : d1);
  return mine;
}

template <class S, bool SUB>
__device__ __forceinline__ void update_site_lanes(const ChainDesc &d, uint32_t sweep, int colour, int mu,
                                                  const SiteGeo &g, uint32_t c0, bool valid, const DrawPre &mine,
                                                  uint32_t &nprop, uint32_t &nacc, float &dr) {
  const int Vh = d.Vh, oc = colour ^ 1, layer = g.layer;
  const int lane = threadIdx.x & 31, l8 = lane & 7, base = lane & 24;
  const int js = g.s >> 1;
  int offp, flp;
  step_fwd(d, sel(g.x, mu), mu, offp, flp);
  const int sp = g.s + offp, lp = lflip<SUB>(d, layer, flp);  // x + mu
  const uint2 key = make_uint2(d.seed_lo, d.seed_hi);

  // this lane's links
  const int ns = 2 * (d.D - 1), t = l8 < ns ? l8 : 0;
  const bool up = (t & 1) == 0;
  int nu = t >> 1;
  nu += nu >= mu ? 1 : 0;
  int offn, fln, offm, flm;
  const int xnu = sel(g.x, nu);
  step_fwd(d, xnu, nu, offn, fln);
  step_bwd(d, xnu, nu, offm, flm);
  const int sn = g.s + offn, ln = lflip<SUB>(d, layer, fln);  // x + nu
  const int sm = g.s + offm, lm = lflip<SUB>(d, layer, flm);  // x - nu
  const int spm = sp + offm, lpm = lflip<SUB>(d, lp, flm);    // x + mu - nu
  // upper: X = U_nu(x), Y = U_mu(x+nu), G = U_nu(x+mu); lower: X = U_mu(x-nu),
  // Y = U_nu(x+mu-nu), G = U_nu(x-nu)
  const M3<float> Y = S::load(up ? plane_ptr<S>(d, ln, oc, mu) : plane_ptr<S>(d, lpm, colour, nu), Vh, (up ? sn : spm) >> 1);
  const M3<float> X = S::load2(up ? plane_ptr<S>(d, layer, colour, nu) : plane_ptr<S>(d, lm, oc, mu), Vh, (up ? g.s : sm) >> 1);
  const M3<float> G = S::load(up ? plane_ptr<S>(d, lp, oc, nu) : plane_ptr<S>(d, lm, oc, nu), Vh, (up ? sp : sm) >> 1);
  M3<float> U = S::load(plane_ptr<S>(d, layer, colour, mu), Vh, js);

  // this lane's staple
  M3<float> M = mul_nn_2(X, Y);
  third_row(M);
  M3<float> P;
  if (up)
    P = mul_nd_2(G, M);
  else
    P = mul_dn_2(M, G);
  M3<float> A = m3_zero<float>();
#pragma unroll
  for (int l = 0; l < 2 * (kMaxD - 1); ++l) {
    if (l >= ns) break;
    M3<float> q;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        q.e[i][j] = {__shfl_sync(0xffffffffu, P.e[i][j].re, base + l), __shfl_sync(0xffffffffu, P.e[i][j].im, base + l)};
    acc_su3_2rows(A, q);
  }

  uint32_t np = 0, na = 0;
  float dretr = 0.0f;
  const float ca = 2.0f * d.beta_f / 3.0f;
#pragma unroll
  for (int sg = 0; sg < 3; ++sg) {
    const int i = (sg == 2) ? 1 : 0;
    const int j = (sg == 0) ? 1 : 2;
    DrawPre pre;
    pre.L = __shfl_sync(0xffffffffu, mine.L, base + sg);
    pre.u4sq = __shfl_sync(0xffffffffu, mine.u4sq, base + sg);
    pre.costh = __shfl_sync(0xffffffffu, mine.costh, base + 3 + sg);
    pre.sinth = __shfl_sync(0xffffffffu, mine.sinth, base + 3 + sg);
    pre.cphi = __shfl_sync(0xffffffffu, mine.cphi, base + 3 + sg);
    pre.sphi = __shfl_sync(0xffffffffu, mine.sphi, base + 3 + sg);
    cm_subgroup_f<true>(U, A, i, j, ca, d.hits, key, c0, sweep, heatbath_tag(colour, mu, sg), pre, np, na, dretr);
    __syncwarp();
  }
  if (!valid) return;
  if (l8 == 0) {
    nprop += np;
    nacc += na;
    dr = dretr;
  }
  for_replicas<SUB>(d, g, l8, 8, [&](int vl, int j) { S::store(plane_ptr<S>(d, vl, colour, mu), Vh, j, U); });
}

// ------------------------------------------------------------------ FP64 link update in fixed point
// The one-coupling FP64 update with its linear algebra (staples, projections,
// rotations) in the integers of su3_fixed.cuh.

// Row `row` of a stored FP64 link in fixed point.
template <bool COH = false>
__device__ __forceinline__ void load_row_f(const StoreF64x18::Vec *plane, int Vh, int jj, int row, Fc (&r)[3],
                                           FxRange &rg) {
  if (!in_bounds(jj, Vh, kBoundsIndex)) {
    r[0] = r[1] = r[2] = Fc{{0, 0}, {0, 0}};
    return;
  }
  const double2 *p = plane + jj + 3 * row * Vh;
  const double2 q0 = ld_link<COH>(p), q1 = ld_link<COH>(p + Vh), q2 = ld_link<COH>(p + 2 * Vh);
  r[0] = fc_of(q0.x, q0.y, rg);
  r[1] = fc_of(q1.x, q1.y, rg);
  r[2] = fc_of(q2.x, q2.y, rg);
}

template <bool COH = false>
__device__ __forceinline__ void load_f(const StoreF64x18::Vec *plane, int Vh, int jj, FM3 &m, FxRange &rg) {
#pragma unroll
  for (int i = 0; i < 3; ++i) load_row_f<COH>(plane, Vh, jj, i, m.e[i], rg);
}

// The draw of one subgroup in double, out of line: proposals with too few
// digits in fixed point only (propose_fx).
struct DrawD {
  double x[4];
  uint32_t nprop;
  bool accepted;
};
static __device__ __noinline__ DrawD su2_draw_general(double alpha, int hits, uint2 key, uint32_t c0, uint32_t c1,
                                               uint32_t tag) {
  DrawD r;
  r.nprop = 0;
  r.accepted = su2_draw_d(alpha, hits, key, c0, c1, tag, r.x, r.nprop);
  return r;
}

// The three links of one staple (staple_f): rows 0, 1 of X, all of Y and G.
// t counts the 2 (D - 1) staples: the upper ones of the other directions in
// order, then the lower ones.
template <bool SUB, bool COH>
__device__ __forceinline__ void staple_fixed(const ChainDesc &d, const SiteGeo &g, int colour, int mu, int t, int sp,
                                             int lp, FSum &A, FxRange &rg) {
  using S = StoreF64x18;
  const int Vh = d.Vh, oc = colour ^ 1, layer = g.layer;
  const bool up = t < d.D - 1;
  int nu = up ? t : t - (d.D - 1);
  nu += nu >= mu ? 1 : 0;
  int offn, fln, offm, flm;
  const int xnu = sel(g.x, nu);
  step_fwd(d, xnu, nu, offn, fln);
  step_bwd(d, xnu, nu, offm, flm);
  const int sn = g.s + offn, ln = lflip<SUB>(d, layer, fln);  // x + nu
  const int sm = g.s + offm, lm = lflip<SUB>(d, layer, flm);  // x - nu
  const int spm = sp + offm, lpm = lflip<SUB>(d, lp, flm);    // x + mu - nu
  const S::Vec *py = up ? plane_ptr<S>(d, ln, oc, mu) : plane_ptr<S>(d, lpm, colour, nu);
  const S::Vec *px = up ? plane_ptr<S>(d, layer, colour, nu) : plane_ptr<S>(d, lm, oc, mu);
  const S::Vec *pg = up ? plane_ptr<S>(d, lp, oc, nu) : plane_ptr<S>(d, lm, oc, nu);
  const int jy = (up ? sn : spm) >> 1, jx = (up ? g.s : sm) >> 1, jg = (up ? sp : sm) >> 1;
  FM3 Y, G;
  Fc X[2][3];
  load_f<COH>(py, Vh, jy, Y, rg);
  load_row_f<COH>(px, Vh, jx, 0, X[0], rg);
  load_row_f<COH>(px, Vh, jx, 1, X[1], rg);
  load_f<COH>(pg, Vh, jg, G, rg);
  staple_f(A, X, Y, G, up, rg);
}

__device__ __forceinline__ Direction direction_of(uint2 w) {
  Direction r;
  int64_t c, s;
  trig_fx(w.y, 1, c, s);
  r.st = sin_theta_fx(w.x);
  r.ct = cos_theta_fx(w.x);
  r.cphi = fx_split(c);
  r.sphi = fx_split(s);
  return r;
}

// The proposals h, h + 1, ... of a subgroup until one is not rejected.
__device__ __forceinline__ ProposalStatus propose_until(int &h, int hits, uint2 key, uint32_t c0, uint32_t c1,
                                                        uint32_t tag, const FxNorm &n, const InvBeta &ib,
                                                        Proposal &p) {
  ProposalStatus st = kRejected;
#pragma unroll 1
  for (; h < hits && st == kRejected; ++h) {
    const uint4 w = philox4x32_10(make_uint4(c0, c1, tag | (uint32_t)h, kPurposeHeatbath), key);
    int64_t cs, sn;
    trig_fx(2u * w.y + 1u, 0, cs, sn);
    st = propose_fx(radius_fx(neg_log_fx(w.x), neg_log_fx(w.z), cs), square_fx(w.w), n, ib, p);
  }
  return st;
}

__device__ __forceinline__ void swap_rows(Fc (&a)[3], Fc (&b)[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const Fc t = a[k];
    a[k] = b[k];
    b[k] = t;
  }
}

// cm_update with U in units 2^-60 and the staple sum in units 2^-56, all in
// fixed point.  The loop over the subgroups stays a loop (its body once in
// the instruction cache): the rows of U and the columns of A of the current
// subgroup are swapped into places 0 and 1.
// dretr2: the change of Re Tr(U A) / 2 in units 2^-57.  nprop negative: a
// norm out of range (norm_fx), nothing of the update is to be used.
__device__ __forceinline__ void cm_update_fixed(const ChainDesc &d, FM3 &U, const FM3 &A, uint32_t c0, uint32_t c1,
                                                int colour, int mu, int32_t &nprop, uint32_t &nacc,
                                                int64_t &dretr2) {
  const uint2 key = make_uint2(d.seed_lo, d.seed_hi);
  const InvBeta ib = {d.inv_beta_m, d.inv_beta_e};
  const int hits = d.hits;
  Fc(&u0)[3] = U.e[0], (&u1)[3] = U.e[1], (&u2)[3] = U.e[2];
  Fc a0[3], a1[3], a2[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    a0[k] = A.e[k][0];
    a1[k] = A.e[k][1];
    a2[k] = A.e[k][2];
  }
  dretr2 = 0;
  uint4 dir = {};  // the direction block: subgroups 0 and 1 share one (direction_words)
#pragma unroll 1
  for (int sg = 0; sg < 3; ++sg) {
    const uint32_t tag = heatbath_tag(colour, mu, sg);
    if (sg != 1) dir = philox4x32_10(make_uint4(c0, c1, tag | kHitDirection, kPurposeHeatbath), key);
    FxAcc s[4] = {{0, kHalf60}, {0, kHalf60}, {0, kHalf60}, {0, kHalf60}};
#pragma unroll
    for (int k = 0; k < 3; ++k) project_k_f(s, u0[k], u1[k], a0[k], a1[k]);
    const int64_t a[4] = {fold60(s[0]), fold60(s[1]), fold60(s[2]), fold60(s[3])};  // 2^-56, and the factor 1/2
    FxNorm n;
    if (norm_fx<true>(a, n, nprop)) {
      Proposal p;
      int h = 0;
      const ProposalStatus st = propose_until(h, hits, key, c0, c1, tag, n, ib, p);
      Fx x[4];
      bool accepted = st == kAccepted;
      if (accepted) {
        direction_fx(p, direction_of(sg == 1 ? make_uint2(dir.z, dir.w) : make_uint2(dir.x, dir.y)), x);
      } else if (st == kInDouble) {
        const DrawD r = su2_draw_general(2.0 * d.beta_d / 3.0 * dbl_of(n.kappa, 57 + n.s), hits, key, c0, c1, tag);
        h = (int)r.nprop;
        accepted = r.accepted;
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = fx_of(r.x[q]);
      }
      nprop += h;
      if (accepted) {
        ++nacc;
        // k x0 - a0 with k = kappa 2^(3 - s)
        dretr2 += shift_round(fx_mul(fx_split(n.kappa), x[0]), n.s) - a[0];
        Fx r[4], rn[4];
        quat_fx(x, n.v, r);
#pragma unroll
        for (int q = 0; q < 4; ++q) rn[q] = fx_neg(r[q]);
#pragma unroll
        for (int k = 0; k < 3; ++k) rotate_col_f(u0[k], u1[k], r, rn);
      }
    }
    // subgroups (0,1), (0,2), (1,2)
    if (sg == 0) {
      swap_rows(u1, u2);
      swap_rows(a1, a2);
    } else if (sg == 1) {  // places hold rows 0, 2, 1
      swap_rows(u0, u2);   // 1, 2, 0
      swap_rows(a0, a2);
    }
  }
}

// The counts and the action change of one update.
struct UpdateCount {
  uint32_t nprop, nacc;
  double dretr;
};

// The double-precision update of one site, out of line: links outside the
// fixed-point range only.
template <bool SUB, bool COH>
__device__ __noinline__ UpdateCount update_site_f64_general(const ChainDesc *d, uint32_t sweep, int colour, int mu,
                                                            int layer, int jj) {
  UpdateCount u = {0, 0, 0.0};
  if constexpr (SUB)
    update_site<StoreF64x18T<COH>, false, false, true>(*d, sweep, colour, mu, layer, jj, u.nprop, u.nacc, u.dretr);
  else
    update_site_lean<StoreF64x18T<COH>, false>(*d, sweep, colour, mu, layer, jj, u.nprop, u.nacc, u.dretr);
  return u;
}

// The change of Re Tr(U A) of one update: rounded to units 2^-51, the last
// place of a double of its size (at most 36 for SU(3) links; sums over a warp
// are exact), and in double where the double-precision form ran.
struct ActionChange {
  int64_t v;
  double general;
};

// One thread per link.
template <bool SUB>
__device__ __forceinline__ void update_site_fixed(const ChainDesc &d, uint32_t sweep, int colour, int mu, int layer,
                                                  int jj, uint32_t &nprop, uint32_t &nacc, ActionChange &dr) {
  using S = StoreF64x18;
  const int Vh = d.Vh;
  const SiteGeo g = site_of<SUB>(d, layer, colour, jj);
  const int js = g.s >> 1;
  int offp, flp;
  step_fwd(d, sel(g.x, mu), mu, offp, flp);
  const int sp = g.s + offp, lp = lflip<SUB>(d, layer, flp);  // x + mu
  FSum A = {};
  FxRange rg;
  // one staple at a time: its instructions once, not six times, in the
  // instruction cache
#pragma unroll 1
  for (int t = 0; t < 2 * (d.D - 1); ++t) staple_fixed<SUB, false>(d, g, colour, mu, t, sp, lp, A, rg);
  S::Vec *pu = plane_ptr<S>(d, layer, colour, mu);
  FM3 U;
  load_f(pu, Vh, js, U, rg);
  int32_t np = -1;
  uint32_t na = 0;
  int64_t half;
  if (rg.ok()) {
    np = 0;
    cm_update_fixed(d, U, factor56(A), site_key<SUB>(d, g), sweep, colour, mu, np, na, half);
  }
  if (np < 0) {
    const UpdateCount u = update_site_f64_general<SUB, false>(&d, sweep, colour, mu, layer, jj);
    nprop += u.nprop;
    nacc += u.nacc;
    dr.general = u.dretr;
    return;
  }
  nprop += (uint32_t)np;
  nacc += na;
  dr.v = shift_round(half, 5);
  // a link none of whose subgroups accepted keeps its bits
  if (na && in_bounds(js, Vh, kBoundsIndex)) {
    // the rows lie in the order 1, 2, 0 after the last subgroup
    double2 v[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const Fc e = U.e[(q / 3 + 2) % 3][q % 3];
      v[q] = make_double2(dbl_of(fx_val(e.re), 60), dbl_of(fx_val(e.im), 60));
    }
    for_replicas<SUB>(d, g, 0, 1, [&](int vl, int j) {
      S::Vec *p = plane_ptr<S>(d, vl, colour, mu) + j;
#pragma unroll
      for (int q = 0; q < 9; ++q) p[q * Vh] = v[q];
    });
  }
}

__device__ __forceinline__ Fx shfl_fx(const Fx &a, int src) {
  return {__shfl_sync(0xffffffffu, a.h, src), __shfl_sync(0xffffffffu, a.l, src)};
}
__device__ __forceinline__ int64_t shfl_ll(int64_t a, int src) { return __shfl_sync(0xffffffffu, (long long)a, src); }
__device__ __forceinline__ int64_t shfl_xor_ll(int64_t a, int m) {
  return __shfl_xor_sync(0xffffffffu, (long long)a, m);
}

// Eight lanes per link, for lattices that do not fill the GPU with one
// thread per link (an update is then one thread's chain of ~20000 dependent
// instructions): each lane forms one staple (integer sums: the same total in
// any order), the logarithms, angles and directions of the three subgroups'
// first proposals take one pass over the lanes, and lanes 0..2 hold one
// column of U each in the projections and rotations.  Results are bitwise
// those of update_site_fixed.  Called by whole warps; lanes without a link
// (valid false) run along on a repeated one.

// Lane l's part of the draws (no link is read).  A block of random words per
// lane (lanes 0..2: the first proposals, 3 and 4: the direction blocks of
// subgroups 0, 1 and of subgroup 2), then lanes 0..2 take ln u1 and the
// proposal's angle, lanes 3..5 ln u3 and the direction.
struct CoopDraws {
  int64_t L, u4sq;        // lanes 0..2
  Fx st, ct, cphi, sphi;  // lanes 3..5
};
__device__ __forceinline__ CoopDraws coop_draws(uint2 key, uint32_t c0, uint32_t sweep, int colour, int mu) {
  const int lane = threadIdx.x & 31, l8 = lane & 7, base = lane & 24;
  const int sub = l8 < 3 ? l8 : (l8 < 6 ? l8 - 3 : 0);
  const uint32_t btag = heatbath_tag(colour, mu, l8 < 3 ? l8 : (l8 == 4 ? 2 : 0)) | (l8 < 3 ? 0u : kHitDirection);
  const uint4 w = philox4x32_10(make_uint4(c0, sweep, btag, kPurposeHeatbath), key);
  const int dl = base + (sub == 2 ? 4 : 3);
  const uint32_t d0 = __shfl_sync(0xffffffffu, w.x, dl), d1 = __shfl_sync(0xffffffffu, w.y, dl);
  const uint32_t d2 = __shfl_sync(0xffffffffu, w.z, dl), d3 = __shfl_sync(0xffffffffu, w.w, dl);
  const uint32_t w3rd = __shfl_sync(0xffffffffu, w.z, base + sub);
  const uint32_t wth = sub == 1 ? d2 : d0, wphi = sub == 1 ? d3 : d1;
  const bool prop = l8 < 3;
  int64_t cs, sn;
  trig_fx(prop ? 2u * w.y + 1u : wphi, prop ? 0 : 1, cs, sn);
  const int64_t nl = neg_log_fx(prop ? w.x : w3rd);
  CoopDraws r;
  r.L = radius_fx(nl, shfl_ll(nl, base + ((l8 + 3) & 7)), cs);
  r.u4sq = square_fx(w.w);
  r.st = sin_theta_fx(wth);
  r.ct = cos_theta_fx(wth);
  r.cphi = fx_split(cs);
  r.sphi = fx_split(sn);
  return r;
}

template <bool SUB, bool COH = false>
__device__ __forceinline__ void update_site_coop(const ChainDesc &d, uint32_t sweep, int colour, int mu,
                                                 const SiteGeo &g, int jj, uint32_t c0, bool valid,
                                                 const CoopDraws &mine, uint32_t &nprop, uint32_t &nacc,
                                                 ActionChange &dr) {
  using S = StoreF64x18;
  const int Vh = d.Vh, layer = g.layer;
  const int lane = threadIdx.x & 31, l8 = lane & 7, base = lane & 24;
  const int js = g.s >> 1;
  int offp, flp;
  step_fwd(d, sel(g.x, mu), mu, offp, flp);
  const int sp = g.s + offp, lp = lflip<SUB>(d, layer, flp);  // x + mu
  const uint2 key = make_uint2(d.seed_lo, d.seed_hi);
  const InvBeta ib = {d.inv_beta_m, d.inv_beta_e};
  const int hits = d.hits;

  // staples
  FSum A = {};
  FxRange rg;
  const int ns = 2 * (d.D - 1);
  staple_fixed<SUB, COH>(d, g, colour, mu, l8 < ns ? l8 : 0, sp, lp, A, rg);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      int64_t re = l8 < ns ? A.re[i][j] : 0, im = l8 < ns ? A.im[i][j] : 0;
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        re += shfl_xor_ll(re, o);
        im += shfl_xor_ll(im, o);
      }
      A.re[i][j] = re;
      A.im[i][j] = im;
    }
  // column c of U, row c of A
  const int c = l8 & 3, cc = c < 3 ? c : 0;
  S::Vec *pu = plane_ptr<S>(d, layer, colour, mu);
  Fc u[3], a[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    double2 q = make_double2(0.0, 0.0);
    if (in_bounds(js, Vh, kBoundsIndex)) q = ld_link<COH>(pu + js + (3 * r + cc) * Vh);
    u[r] = fc_of(q.x, q.y, rg);
    const int64_t re = cc == 0 ? A.re[0][r] : (cc == 1 ? A.re[1][r] : A.re[2][r]);
    const int64_t im = cc == 0 ? A.im[0][r] : (cc == 1 ? A.im[1][r] : A.im[2][r]);
    a[r] = {fx_split((re + 8) >> 4), fx_split((im + 8) >> 4)};
    if (c == 3) u[r] = a[r] = Fc{{0, 0}, {0, 0}};
  }
  const bool bad = (__ballot_sync(0xffffffffu, !rg.ok()) >> base & 0xffu) != 0;

  uint32_t np = 0, na = 0;
  int64_t half = 0;
  int32_t large = 0;
#pragma unroll 1
  for (int sg = 0; sg < 3; ++sg) {
    // the projection: this lane's k, then the sum over the lanes (the rounding
    // constant enters once)
    const int64_t round = c == 0 ? kHalf60 : 0;
    FxAcc s[4] = {{0, round}, {0, round}, {0, round}, {0, round}};
    project_k_f(s, u[0], u[1], a[0], a[1]);
    int64_t pa[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        s[q].hh += shfl_xor_ll(s[q].hh, o);
        s[q].x += shfl_xor_ll(s[q].x, o);
      }
      pa[q] = fold60(s[q]);
    }
    const int64_t L = shfl_ll(mine.L, base + sg), u4 = shfl_ll(mine.u4sq, base + sg);
    Direction dir;
    dir.st = shfl_fx(mine.st, base + 3 + sg);
    dir.ct = shfl_fx(mine.ct, base + 3 + sg);
    dir.cphi = shfl_fx(mine.cphi, base + 3 + sg);
    dir.sphi = shfl_fx(mine.sphi, base + 3 + sg);
    FxNorm n;
    if (norm_fx<false>(pa, n, large)) {
      const uint32_t tag = heatbath_tag(colour, mu, sg);
      Proposal p;
      int h = 1;
      ProposalStatus st = propose_fx(L, u4, n, ib, p);
      if (st == kRejected) st = propose_until(h, hits, key, c0, sweep, tag, n, ib, p);
      Fx x[4];
      bool accepted = st == kAccepted;
      if (accepted) {
        direction_fx(p, dir, x);
      } else if (st == kInDouble) {
        const DrawD r = su2_draw_general(2.0 * d.beta_d / 3.0 * dbl_of(n.kappa, 57 + n.s), hits, key, c0, sweep, tag);
        h = (int)r.nprop;
        accepted = r.accepted;
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = fx_of(r.x[q]);
      }
      np += (uint32_t)h;
      if (accepted) {
        ++na;
        half += shift_round(fx_mul(fx_split(n.kappa), x[0]), n.s) - pa[0];
        Fx r[4], rn[4];
        quat_fx(x, n.v, r);
#pragma unroll
        for (int q = 0; q < 4; ++q) rn[q] = fx_neg(r[q]);
        rotate_col_f(u[0], u[1], r, rn);
      }
    }
    __syncwarp();
    // subgroups (0,1), (0,2), (1,2): as cm_update_fixed
    const int keep = sg == 0 ? 0 : 1;
    const Fc tu = u[2], ta = a[2];
    u[2] = fc_sel(keep == 0, u[1], u[0]);
    a[2] = fc_sel(keep == 0, a[1], a[0]);
    u[0] = fc_sel(keep == 0, u[0], tu);
    a[0] = fc_sel(keep == 0, a[0], ta);
    u[1] = fc_sel(keep == 0, tu, u[1]);
    a[1] = fc_sel(keep == 0, ta, a[1]);
  }
  if (!valid) return;
  if (bad || large < 0) {  // the same in a link's lanes
    if (l8 == 0) {
      const UpdateCount uc = update_site_f64_general<SUB, COH>(&d, sweep, colour, mu, layer, jj);
      nprop += uc.nprop;
      nacc += uc.nacc;
      dr.general = uc.dretr;
    }
    return;
  }
  if (l8 == 0) {
    nprop += np;
    nacc += na;
    dr.v = shift_round(half, 5);
  }
  // after the last swap the rows lie in the order 0, 2, 1
  if (l8 < 3 && na && in_bounds(js, Vh, kBoundsIndex)) {
    double2 v[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const Fc e = u[r == 0 ? 0 : 3 - r];
      v[r] = make_double2(dbl_of(fx_val(e.re), 60), dbl_of(fx_val(e.im), 60));
    }
    for_replicas<SUB>(d, g, 0, 1, [&](int vl, int j) {
      S::Vec *p = plane_ptr<S>(d, vl, colour, mu) + j + c * Vh;
#pragma unroll
      for (int r = 0; r < 3; ++r) p[3 * r * Vh] = v[r];
    });
  }
}

// ------------------------------------------------------------------ re-unitarisation

__device__ __forceinline__ double to_double(float x) { return f2d_bits(x); }
__device__ __forceinline__ double to_double(double x) { return x; }

// Rows 1, 2 of a stored link in double (row 3 is rebuilt by reunit_d, or
// not kept at all by two-row storage).
template <class S>
__device__ __forceinline__ M3<double> load_rows2_d(const typename S::Vec *p, int Vh, int js) {
  const M3<typename S::R> f = S::load2(p, Vh, js);
  M3<double> m;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      m.e[i][j] = i < 2 ? C<double>{to_double(f.e[i][j].re), to_double(f.e[i][j].im)} : C<double>{0.0, 0.0};
  return m;
}

// The end of reunit_rows2_f: the corrections applied in float.
__device__ __forceinline__ void reunit_apply_f(M3<float> &m, float e1, float pr, float pi, float e2) {
  C<float> *r1 = m.e[0], *r2 = m.e[1];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const C<float> a = r1[k];
    r1[k] = {fm(a.re, e1, a.re), fm(a.im, e1, a.im)};
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    // c = -p r1'_k, then r2''_k = r2_k + (c (1 + e2) + r2_k e2), one rounding
    const C<float> a = r1[k], b = r2[k];
    const float cr = fm(pi, a.im, -pr * a.re), ci = fm(-pi, a.re, -pr * a.im);
    r2[k] = {b.re + fm(b.re, e2, fm(cr, e2, cr)), b.im + fm(b.im, e2, fm(ci, e2, ci))};
  }
}

// The double-precision Gram-Schmidt of two float rows r1, r2, applied in
// float.  The norms and the inner product are summed in double from the
// float elements (products of floats are exact in double):
//   n1 = |r1|^2, s1 = n1^(-1/2), q = <r1, r2>, p = s1 q = <r1', r2>,
//   n2 = |r2 - p r1'|^2 = |r2|^2 - |p|^2 (as |r1'| = 1), s2 = n2^(-1/2).
// The results r1' = r1 s1 and r2'' = (r2 - p r1') s2 differ from the stored
// rows by corrections of the rows' departure from orthonormality (~1e-7
// between re-unitarisations): r1' = r1 + r1 e1 with e1 = s1 - 1, and
// r2'' = r2 + (c (1 + e2) + r2 e2) with c = -p r1' and e2 = s2 - 1.  Each
// correction is formed in float (the factors e1, p, e2 rounded to float:
// relative errors 2^-24 of small quantities) and added with a single
// rounding, so the stored floats are the double computation's rounded
// result except where that result lies within ~1e-14 of a rounding boundary
// (1e-12 for departures of 1e-4).  38 double operations per link instead of
// 56, on a pipe that runs at 1/64 of the float rate here.
__device__ __forceinline__ void reunit_rows2_f(M3<float> &m) {
  C<float> *r1 = m.e[0], *r2 = m.e[1];
  double n1 = f2d_bits(r1[0].re) * f2d_bits(r1[0].re);
  n1 = fm(f2d_bits(r1[0].im), f2d_bits(r1[0].im), n1);
  double n2 = f2d_bits(r2[0].re) * f2d_bits(r2[0].re);
  n2 = fm(f2d_bits(r2[0].im), f2d_bits(r2[0].im), n2);
  // q = sum_k conj(r1_k) r2_k
  double qr = f2d_bits(r1[0].re) * f2d_bits(r2[0].re), qi = f2d_bits(r1[0].re) * f2d_bits(r2[0].im);
  qr = fm(f2d_bits(r1[0].im), f2d_bits(r2[0].im), qr);
  qi = fm(-f2d_bits(r1[0].im), f2d_bits(r2[0].re), qi);
#pragma unroll
  for (int k = 1; k < 3; ++k) {
    const double ar = f2d_bits(r1[k].re), ai = f2d_bits(r1[k].im), br = f2d_bits(r2[k].re), bi = f2d_bits(r2[k].im);
    n1 = fm(ar, ar, n1);
    n1 = fm(ai, ai, n1);
    n2 = fm(br, br, n2);
    n2 = fm(bi, bi, n2);
    qr = fm(ar, br, qr);
    qr = fm(ai, bi, qr);
    qi = fm(ar, bi, qi);
    qi = fm(-ai, br, qi);
  }
  const double s1 = rsqrt_d<1>(n1);
  const double pdr = s1 * qr, pdi = s1 * qi;
  n2 = fm(-pdr, pdr, n2);
  n2 = fm(-pdi, pdi, n2);
  const double s2 = rsqrt_d<1>(n2);
  reunit_apply_f(m, d2f_bits(s1 - 1.0), d2f_bits(pdr), d2f_bits(pdi), d2f_bits(s2 - 1.0));
}

// reunit_apply_f, and whether its floats are sure to be those of the
// double-precision factors too: those differ from the factors given here
// (exact to 2^-57) by up to 1e-15, so each result must not change when its
// correction moves by that and by two ulps.
__device__ __forceinline__ bool reunit_apply_sure(M3<float> &m, float e1, float pr, float pi, float e2) {
  constexpr float kAbs = 4e-15f, kRel = 0x1p-22f;
  C<float> *r1 = m.e[0], *r2 = m.e[1];
  const float eta1 = fm(fabsf(e1), kRel, kAbs), lo = e1 - eta1, hi = e1 + eta1;
  bool sure = true;
  const auto first = [&](float a) {
    sure = sure && fm(a, lo, a) == fm(a, hi, a);
    return fm(a, e1, a);
  };
  const auto second = [&](float b, float c) {
    const float corr = fm(b, e2, fm(c, e2, c)), eta = fm(fabsf(corr), kRel, kAbs);
    sure = sure && b + (corr - eta) == b + (corr + eta);
    return b + corr;
  };
#pragma unroll
  for (int k = 0; k < 3; ++k) r1[k] = {first(r1[k].re), first(r1[k].im)};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const C<float> a = r1[k];
    r2[k] = {second(r2[k].re, fm(pi, a.im, -pr * a.re)), second(r2[k].im, fm(-pi, a.re, -pr * a.im))};
  }
  return sure;
}

// One stored link in double precision, out of line: links whose rows are far
// from orthonormal, or whose float rounding is not sure (reunit_link).
template <class S>
static __device__ __noinline__ void reunit_link_general(typename S::Vec *p, int Vh, int js) {
  if constexpr (S::kTwoRows) {
    M3<float> m = S::load2(p, Vh, js);
    reunit_rows2_f(m);
    S::store(p, Vh, js, m);
  } else {
    constexpr int kNewton = sizeof(typename S::R) == 4 ? 1 : 2;  // float storage: one Newton step suffices
    M3<double> m = load_rows2_d<S>(p, Vh, js);
    reunit_d<kNewton, true>(m);
    S::store(p, Vh, js, to_storage<typename S::R>(m));
  }
}

// Re-unitarise one stored link: the sums, products and reciprocal square roots
// in fixed point (errors below 2^-57, absolute; the double-precision pipe ran
// at 90 % of its rate here), the result rounded to the storage precision, or
// applied to two-row float storage as in reunit_rows2_f.  Float links that
// might round differently from the double-precision form (one warp in
// several hundred holds such a link; links with zeros always) take that form:
// the stored floats are its floats.
template <class S>
__device__ __forceinline__ void reunit_link(typename S::Vec *p, int Vh, int js) {
  using R = typename S::R;
  M3<R> m = S::load2(p, Vh, js);
  FxRange rg;
  FM3 f;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if constexpr (sizeof(R) == 4) {
        rg.doubles(__float_as_int(m.e[i][k].re), __float_as_int(m.e[i][k].im));
        f.e[i][k] = {fx_of(m.e[i][k].re), fx_of(m.e[i][k].im)};
      } else {
        rg.doubles(dbl_hi(m.e[i][k].re), dbl_hi(m.e[i][k].im));
        f.e[i][k] = {fx_of_pipe(m.e[i][k].re), fx_of_pipe(m.e[i][k].im)};
      }
    }
  const bool in = rg.ok(sizeof(R) == 4 ? kElemMaxFloat : kElemMaxHi);
  FxRange rr;
  if constexpr (S::kTwoRows) {
    float e1, pr, pi, e2;
    if (in && reunit_factors_f(f.e[0], f.e[1], e1, pr, pi, e2)) {
      if (reunit_apply_sure(m, e1, pr, pi, e2)) {
        S::store(p, Vh, js, m);
        return;
      }
    }
  } else if (in && reunit_f<sizeof(R) == 4>(f, rr) && rr.ok()) {
    bool sure = true;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int64_t re = fx_val(f.e[i][k].re), im = fx_val(f.e[i][k].im);
        if constexpr (sizeof(R) == 4) {
          m.e[i][k].re = flt_of_sure(re, sure);
          m.e[i][k].im = flt_of_sure(im, sure);
        } else
          m.e[i][k] = {dbl_of_pipe(re, 60), dbl_of_pipe(im, 60)};
      }
    if (sure) {
      S::store(p, Vh, js, m);
      return;
    }
  }
  reunit_link_general<S>(p, Vh, js);
}

// All links of the two sites of a checkerboard index (many-chain launches).
template <class S>
__device__ __forceinline__ void reunit_site(const ChainDesc &d, int layer, int jj) {
#pragma unroll 1
  for (int cm = 0; cm < 2 * d.D; ++cm)
    reunit_link<S>(plane_ptr<S>(d, layer, cm / d.D, cm % d.D), d.Vh, jj);
}

// ------------------------------------------------------------------ measurements
// Sums in double: plaquettes split space/time, and Polyakov lines started at
// x^D = 0.

// Re Tr(U_mu(x) U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+) = Re Tr(P Q^+) with
// P = U_mu(x) U_nu(x+mu), Q = U_nu(x) U_mu(x+nu), both in SU(3): rows 1, 2
// of P and Q come from rows 1, 2 of U_mu(x) and U_nu(x) (um2, un2) and the
// full U_nu(x+mu), U_mu(x+nu); their third rows contribute
// sum_j P_3j conj(Q_3j) = <P_1 x P_2, Q_1 x Q_2> = G_11 G_22 - G_12 G_21
// (the Binet-Cauchy identity; row 3 of an SU(3) matrix is the conjugated
// cross product of rows 1, 2) with G_kl = <P_k, Q_l> = sum_j conj(P_kj) Q_lj.
// The factor 1/3 is applied to the sums.
template <class S, bool SUB = false>
__device__ __forceinline__ typename S::R plaquette_at(const ChainDesc &d, const SiteGeo &g, int colour, int mu, int nu,
                                                      int xmu, int xnu, const M3<typename S::R> &um2) {
  using R = typename S::R;
  const int Vh = d.Vh, layer = g.layer, jj = g.s >> 1, oc = colour ^ 1;
  int offp, flp, offn, fln;
  step_fwd(d, xmu, mu, offp, flp);
  step_fwd(d, xnu, nu, offn, fln);
  const M3<R> a = S::load(plane_ptr<S>(d, lflip<SUB>(d, layer, flp), oc, nu), Vh, (g.s + offp) >> 1);  // U_nu(x+mu)
  const M3<R> b = S::load(plane_ptr<S>(d, lflip<SUB>(d, layer, fln), oc, mu), Vh, (g.s + offn) >> 1);  // U_mu(x+nu)
  const M3<R> un2 = S::load2(plane_ptr<S>(d, layer, colour, nu), Vh, jj);                // U_nu(x), rows 1, 2
  const M3<R> P = mul_nn_2(um2, a), Q = mul_nn_2(un2, b);
  C<R> G[2][2];
#pragma unroll
  for (int k = 0; k < 2; ++k)
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      C<R> x = cmul_cn(P.e[k][0], Q.e[l][0]);
      cmac_cn(x, P.e[k][1], Q.e[l][1]);
      cmac_cn(x, P.e[k][2], Q.e[l][2]);
      G[k][l] = x;
    }
  R tr = G[0][0].re + G[1][1].re;
  tr = fm(G[0][0].re, G[1][1].re, tr);
  tr = fm(-G[0][0].im, G[1][1].im, tr);
  tr = fm(-G[0][1].re, G[1][0].re, tr);
  tr = fm(G[0][1].im, G[1][0].im, tr);
  return tr;
}

// plaquette_at for FP64 links in fixed point: Re Tr in units 2^-60, one
// plaquette at a time (mu, nu are run-time values: the code is short).
// false: a link is out of the fixed-point range.
template <bool SUB>
__device__ __forceinline__ bool plaquette_fixed(const ChainDesc &d, const SiteGeo &g, int colour, int mu, int nu,
                                                int64_t &tr) {
  using S = StoreF64x18;
  const int Vh = d.Vh, layer = g.layer, js = g.s >> 1, oc = colour ^ 1;
  int offp, flp, offn, fln;
  step_fwd(d, sel(g.x, mu), mu, offp, flp);
  step_fwd(d, sel(g.x, nu), nu, offn, fln);
  const S::Vec *pm = plane_ptr<S>(d, layer, colour, mu), *pn = plane_ptr<S>(d, layer, colour, nu);
  FxRange rg;
  FM3 Y, P, Q;
  Fc row[3];
  load_f(plane_ptr<S>(d, lflip<SUB>(d, layer, flp), oc, nu), Vh, (g.s + offp) >> 1, Y, rg);  // U_nu(x+mu)
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    load_row_f(pm, Vh, js, i, row, rg);
    row_nn_f(P, i, row, Y, rg);
  }
  load_f(plane_ptr<S>(d, lflip<SUB>(d, layer, fln), oc, mu), Vh, (g.s + offn) >> 1, Y, rg);  // U_mu(x+nu)
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    load_row_f(pn, Vh, js, i, row, rg);
    row_nn_f(Q, i, row, Y, rg);
  }
  tr = trace_nd_f(P, Q, rg);
  return rg.ok();
}

// The same in double, out of line.
template <bool SUB>
static __device__ __noinline__ double plaquette_general(const ChainDesc *d, int layer, int colour, int jj, int mu,
                                                        int nu) {
  using S = StoreF64x18;
  const SiteGeo g = site_of<SUB>(*d, layer, colour, jj);
  return plaquette_at<S, SUB>(*d, g, colour, mu, nu, sel(g.x, mu), sel(g.x, nu),
                              S::load2(plane_ptr<S>(*d, layer, colour, mu), d->Vh, g.s >> 1));
}

// Sums of plaquettes: integers in units 2^-56 (a site's planes: six at most, of
// magnitude below 7 for links in range), read as one double; and in double
// those of links out of range.
struct PlaquetteSum {
  int64_t v = 0;
  double general = 0.0;
  __device__ __forceinline__ double value() const { return dbl_of(v, 56) + general; }
};

template <bool SUB>
__device__ __forceinline__ void add_plaquette(const ChainDesc &d, const SiteGeo &g, int colour, int jj, int mu, int nu,
                                              PlaquetteSum &s) {
  int64_t tr;
  if (plaquette_fixed<SUB>(d, g, colour, mu, nu, tr))
    s.v += shift_round(tr, 4);
  else
    s.general += plaquette_general<SUB>(&d, g.layer, colour, jj, mu, nu);
}

// The plaquettes of one site: Re Tr summed in the storage precision, split
// into space-like and time-like (the 1/3 is applied with the counts).  The
// loop over mu is unrolled so that the loads of several plaquettes are in
// flight together.  SUB: reads the forward halos.
template <class S, bool SUB = false>
__device__ __forceinline__ void site_plaquettes(const ChainDesc &d, const SiteGeo &g, int colour,
                                                typename S::R &ps, typename S::R &pt) {
  using R = typename S::R;
  const int Vh = d.Vh, D = d.D;
  ps = R(0);
  pt = R(0);
#pragma unroll
  for (int mu = 0; mu + 1 < kMaxD; ++mu) {
    if (mu + 1 >= D) continue;
    const int xmu = sel(g.x, mu);
    const M3<R> um2 = S::load2(plane_ptr<S>(d, g.layer, colour, mu), Vh, g.s >> 1);  // U_mu(x), rows 1, 2
#pragma unroll
    for (int nu = 1; nu < kMaxD; ++nu) {
      if (nu <= mu || nu >= D) continue;
      const R p = plaquette_at<S, SUB>(d, g, colour, mu, nu, xmu, g.x[nu], um2);
      if (nu == D - 1) pt += p; else ps += p;
    }
  }
}

// The same with eight lanes per site: lane p takes plane p (its indices are
// run-time values), the sums are taken in the order of site_plaquettes.
// Called by whole warps; valid false: the lane's site is a repeated one.
template <class S, bool SUB = false>
__device__ __forceinline__ void site_plaquettes_split(const ChainDesc &d, const SiteGeo &g, int colour,
                                                      typename S::R &ps, typename S::R &pt) {
  using R = typename S::R;
  const int D = d.D, lane = threadIdx.x & 31, l8 = lane & 7, base = lane & 24;
  const int np = D * (D - 1) / 2;
  int mu = 0, nu = l8 < np ? l8 + 1 : 1;  // planes (0,1), (0,2), .., (1,2), ..
  while (nu >= D) {
    nu -= D - 2 - mu;
    ++mu;
  }
  const R p = plaquette_at<S, SUB>(d, g, colour, mu, nu, sel(g.x, mu), sel(g.x, nu),
                                   S::load2(plane_ptr<S>(d, g.layer, colour, mu), d.Vh, g.s >> 1));
  ps = R(0);
  pt = R(0);
  int k = 0;
  for (int m = 0; m + 1 < D; ++m)
    for (int n = m + 1; n < D; ++n, ++k) {
      const R q = __shfl_sync(0xffffffffu, p, base + k);
      if (n == D - 1) pt += q; else ps += q;
    }
}

// Tr of the Polyakov line through a site with x^D = 0 (the line follows the
// forward time neighbour until it closes): rows 1, 2 of the running product
// (SU(3)), the next link's load issued before the product.  SUB: only when
// time is undivided (the line then stays inside its box).
template <class S, bool SUB = false>
__device__ __forceinline__ C<typename S::R> polyakov_line(const ChainDesc &d, const SiteGeo &g, int colour) {
  using R = typename S::R;
  const int Vh = d.Vh, t = d.D - 1, layer = g.layer;
  M3<R> P = S::load2(plane_ptr<S>(d, layer, colour, t), Vh, g.s >> 1);
  int cs = g.s, cl = layer, cc = colour, xt = 0;
  auto advance = [&]() {
    int off, fl;
    step_fwd(d, xt, t, off, fl);
    cs += off;
    cl = lflip<SUB>(d, cl, fl);
    cc ^= 1;
    xt = (xt == d.dims[t] - 1) ? 0 : xt + 1;
    return !(cs == g.s && cl == layer);
  };
  bool more = advance();
  M3<R> nxt = more ? S::load(plane_ptr<S>(d, cl, cc, t), Vh, cs >> 1) : m3_zero<R>();
#pragma unroll 1
  while (more) {
    const M3<R> cur = nxt;
    more = advance();
    if (more) nxt = S::load(plane_ptr<S>(d, cl, cc, t), Vh, cs >> 1);
    P = mul_nn_2(P, cur);
  }
  // trace: P_11 + P_22 + P_33 with P_33 = conj(P_11 P_22 - P_12 P_21)
  const C<R> p33 = conj_cross(P.e[0][0], P.e[1][1], P.e[0][1], P.e[1][0]);
  return {P.e[0][0].re + P.e[1][1].re + p33.re, P.e[0][0].im + P.e[1][1].im + p33.im};
}

// The same for FP64 links in fixed point (units 2^-60); false: out of range.
template <bool SUB>
__device__ __forceinline__ bool polyakov_fixed(const ChainDesc &d, const SiteGeo &g, int colour, int64_t &re,
                                               int64_t &im) {
  using S = StoreF64x18;
  const int Vh = d.Vh, t = d.D - 1, layer = g.layer;
  FxRange rg;
  FM3 P, Y;
  load_row_f(plane_ptr<S>(d, layer, colour, t), Vh, g.s >> 1, 0, P.e[0], rg);
  load_row_f(plane_ptr<S>(d, layer, colour, t), Vh, g.s >> 1, 1, P.e[1], rg);
  int cs = g.s, cl = layer, cc = colour, xt = 0;
#pragma unroll 1
  while (true) {
    int off, fl;
    step_fwd(d, xt, t, off, fl);
    cs += off;
    cl = lflip<SUB>(d, cl, fl);
    cc ^= 1;
    xt = (xt == d.dims[t] - 1) ? 0 : xt + 1;
    if (cs == g.s && cl == layer) break;
    load_f(plane_ptr<S>(d, cl, cc, t), Vh, cs >> 1, Y, rg);
    FM3 N;
#pragma unroll
    for (int i = 0; i < 2; ++i) row_nn_f(N, i, P.e[i], Y, rg);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) P.e[i][k] = N.e[i][k];
  }
  // conj(P_11 P_22 - P_12 P_21)
  FxAcc x = {0, kHalf60}, y = {0, kHalf60};
  const Fc r = P.e[0][1];
  cross_f(x, y, P.e[0][0], fx_neg(P.e[0][0].im), P.e[1][1], r, fx_neg(r.re), fx_neg(r.im), P.e[1][0]);
  re = fx_val(P.e[0][0].re) + fx_val(P.e[1][1].re) + fold60(x);
  im = fx_val(P.e[0][0].im) + fx_val(P.e[1][1].im) - fold60(y);
  return rg.ok();
}

template <bool SUB>
static __device__ __noinline__ C<double> polyakov_general(const ChainDesc *d, int layer, int colour, int jj) {
  return polyakov_line<StoreF64x18, SUB>(*d, site_of<SUB>(*d, layer, colour, jj), colour);
}

// A line's trace in double.
template <class S, bool SUB = false>
__device__ __forceinline__ C<double> line_trace(const ChainDesc &d, const SiteGeo &g, int colour, int jj) {
  if constexpr (std::is_same<S, StoreF64x18>::value) {
    int64_t re, im;
    if (polyakov_fixed<SUB>(d, g, colour, re, im)) return {dbl_of(re, 60), dbl_of(im, 60)};
    return polyakov_general<SUB>(&d, g.layer, colour, jj);
  } else {
    const C<typename S::R> l = polyakov_line<S, SUB>(d, g, colour);
    return {to_double(l.re), to_double(l.im)};
  }
}

// Per thread: the two sites of checkerboard index jj (both colours), and the
// Polyakov lines that start at them; accumulated in double.
template <class S>
__device__ __forceinline__ void measure_site(const ChainDesc &d, int layer, int jj, double acc[kPartVals]) {
  using R = typename S::R;
#pragma unroll 1
  for (int colour = 0; colour < 2; ++colour) {
    const SiteGeo g = site_of<false>(d, layer, colour, jj);
    if constexpr (std::is_same<S, StoreF64x18>::value) {
      PlaquetteSum ps, pt;
#pragma unroll 1
      for (int mu = 0; mu + 1 < d.D; ++mu)
#pragma unroll 1
        for (int nu = mu + 1; nu < d.D; ++nu) add_plaquette<false>(d, g, colour, jj, mu, nu, nu == d.D - 1 ? pt : ps);
      acc[0] += ps.value();
      acc[1] += pt.value();
    } else {
      R ps, pt;
      site_plaquettes<S>(d, g, colour, ps, pt);
      acc[0] += to_double(ps);
      acc[1] += to_double(pt);
    }
    if (sel(g.x, d.D - 1) == 0) {
      const C<double> l = line_trace<S>(d, g, colour, jj);
      acc[2] += l.re;
      acc[3] += l.im;
    }
  }
}

// Block reduction of kPartVals doubles in a fixed order.  Result valid in
// thread 0.  Within a warp the four values are spread over the lanes while
// they are summed (six additions instead of twenty: a double addition takes
// 16 clocks of the SM per warp); then warp 0 sums the warps (at most eight).
__device__ __forceinline__ void block_reduce(double v[kPartVals], double *smem /* [32] */) {
  static_assert(kPartVals == 4, "the value index is two lane bits");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  const bool b1 = lane & 16, b0 = lane & 8;
  double x0 = b1 ? v[2] : v[0], x1 = b1 ? v[3] : v[1];
  x0 += __shfl_xor_sync(0xffffffffu, b1 ? v[0] : v[2], 16);
  x1 += __shfl_xor_sync(0xffffffffu, b1 ? v[1] : v[3], 16);
  double x = b0 ? x1 : x0;
  x += __shfl_xor_sync(0xffffffffu, b0 ? x0 : x1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  if ((lane & 7) == 0) smem[warp * kPartVals + (b1 ? 2 : 0) + (b0 ? 1 : 0)] = x;
  __syncthreads();
  if (warp == 0) {
    double y = lane < nw * kPartVals ? smem[lane] : 0.0;
#pragma unroll
    for (int o = kPartVals; o < 32; o <<= 1)
      if (o < nw * kPartVals) y += __shfl_xor_sync(0xffffffffu, y, o);
#pragma unroll
    for (int k = 0; k < kPartVals; ++k) v[k] = __shfl_sync(0xffffffffu, y, k);
  }
  __syncthreads();
}

// Value k of [total, space, time, poly_re, poly_im] from the sums over
// `layers` layers (they hold Re Tr and Tr: the counts carry the factor 3).
__device__ __forceinline__ double measured_value(const ChainDesc &d, const double v[kPartVals], double layers, int k) {
  const int D = d.D;
  const double np_s = 3.0 * d.V * (D - 1) * (D - 2) / 2, np_t = 3.0 * d.V * (D - 1);
  // Polyakov lines are not taken inside sublattice boxes with divided time:
  // the values are NaN
  const double nl = d.hpad[D - 1] ? __longlong_as_double(0x7ff8000000000000ll) : 3.0 * d.spatial_per_layer;
  const double num = k == 0 ? v[0] + v[1] : (k == 1 ? v[0] : (k == 2 ? v[1] : (k == 3 ? v[2] : v[3])));
  const double den = k == 0 ? np_s + np_t : (k == 1 ? np_s : (k == 2 ? np_t : nl));
  return k == 1 && !(np_s > 0) ? 0.0 : num / (layers * den);
}

// Sum the tile partials of one chain per layer (one warp, fixed order) and
// write the values of each layer and of the whole.
__device__ __forceinline__ void finalize_measure(const ChainDesc &d, const double *partials, double *out) {
  const int lane = threadIdx.x & 31;
  double whole[kPartVals] = {0, 0, 0, 0};
  for (int layer = 0; layer < d.nlayers; ++layer) {
    double v[kPartVals] = {0, 0, 0, 0};
    for (int t = lane; t < d.tiles_per_layer; t += 32)
#pragma unroll
      for (int k = 0; k < kPartVals; ++k) v[k] += __ldcg(partials + (size_t)(layer * d.tiles_per_layer + t) * kPartVals + k);
#pragma unroll
    for (int k = 0; k < kPartVals; ++k) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
      v[k] = __shfl_sync(0xffffffffu, v[k], 0);
      whole[k] += v[k];
    }
    if (lane < kMeasVals) out[layer * kMeasVals + lane] = measured_value(d, v, 1.0, lane);
  }
  if (lane < kMeasVals) out[d.nlayers * kMeasVals + lane] = measured_value(d, whole, (double)d.nlayers, lane);
}

// The action bookkeeping restarts at this measurement (a chain whose links
// were replaced asks for it): the measurement becomes the reference and
// the booked changes restart from zero.  Warp-collective; the measurement
// was written by lanes of this warp.
__device__ __forceinline__ void restart_bookkeeping(const ChainDesc &d, const double *out) {
  __syncwarp();
  const int lane = threadIdx.x & 31;
  for (int i = lane; i < (d.nlayers + 1) * kMeasVals; i += 32) d.ref_meas[i] = out[i];
  for (int i = lane; i < d.n_action_slots; i += 32) d.action_slots[i] = 0.0;
}

// ------------------------------------------------------------------ halos

// Entry `e` of the halo list: the links of one halo site of box vl, copied from the site that owns them (the same padded site of
// the neighbouring box given by the entry's offset code, whose box coordinate
// wraps periodically; a wrap across a glued boundary of the double-layered
// torus lands in the other layer).  Halo sites are never sources, so the
// copies do not race.
template <class S>
__device__ __forceinline__ void halo_copy(const ChainDesc &d, int vl, int e) {
  const int4 h = d.halo[e];
  const int colour = e < d.halo_n[0] ? 0 : 1, L = vl / d.nb;
  int bsrc = 0, bmul = 1, flip = 0, rest = vl - L * d.nb;
#pragma unroll
  for (int k = 0; k < kMaxD; ++k)
    if (k < d.D) {
      const int code = (h.z >> (2 * k)) & 3, bc = rest % d.bdiv[k];
      rest /= d.bdiv[k];
      int o = bc + (code == 1 ? -1 : (code == 2 ? 1 : 0));
      if (o < 0 || o >= d.bdiv[k]) {
        o = o < 0 ? o + d.bdiv[k] : o - d.bdiv[k];
        if (d.nlayers == 2) flip ^= (d.glue_mask >> k) & 1;
      }
      bsrc += o * bmul;
      bmul *= d.bdiv[k];
    }
  const int vsrc = (L ^ flip) * d.nb + bsrc;
  for (int mu = 0; mu < d.D; ++mu)
    S::copy(plane_ptr<S>(d, vl, colour, mu), d.Vh, h.x >> 1, plane_ptr<S>(d, vsrc, colour, mu), d.Vh, h.y >> 1);
}

// Warp-sum the FHKP counters and add them to the chain's totals (one of
// kCounterSlots pairs: warps that end together meet on different addresses).
__device__ __forceinline__ void flush_counters(const ChainDesc &d, uint32_t &np, uint32_t &na) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    np += __shfl_down_sync(0xffffffffu, np, o);
    na += __shfl_down_sync(0xffffffffu, na, o);
  }
  if ((threadIdx.x & 31) == 0 && np) {
    unsigned long long *c = d.counters + 2 * (blockIdx.x % kCounterSlots);
    atomicAdd(c + 0, (unsigned long long)np);
    atomicAdd(c + 1, (unsigned long long)na);
  }
  np = 0;
  na = 0;
}

// Register variants of the update kernels: __launch_bounds__(threads, CTAs per
// SM) caps registers at 65536 / (threads x CTAs).  The autotuner times them.
// kRolled: the update keeps its loop over staple directions rolled.
// On the 32^4 workload (one update phase, fresh re-unitarised lattice per
// shape) the best shapes are within 5 % of each other: 128 registers at
// 16 warps per SM is fastest; 96 and 85 registers (spills) are 3-10 % and
// the unconstrained 156 registers (12 warps) 14 % slower.  Dropped after
// measuring: a split into a staple kernel and a heatbath kernel (30 %
// slower), an L1 prefetch of the next staple direction's links (8 %).
template <int V> struct TickBounds;
constexpr int kCoopVariant = 11, kLanesVariant = 12;
template <> struct TickBounds<0> { static constexpr int kThreads = 256, kMinBlocks = 2; static constexpr bool kRolled = false; };   // FP32, 128 regs
template <> struct TickBounds<1> { static constexpr int kThreads = 128, kMinBlocks = 5; static constexpr bool kRolled = false; };   // FP32, 96 regs
template <> struct TickBounds<2> { static constexpr int kThreads = 128, kMinBlocks = 5; static constexpr bool kRolled = true; };    // FP32, rolled, 96 regs
template <> struct TickBounds<3> { static constexpr int kThreads = 256, kMinBlocks = 2; static constexpr bool kRolled = true; };    // FP32, rolled, 128 regs
template <> struct TickBounds<4> { static constexpr int kThreads = 256, kMinBlocks = 3; static constexpr bool kRolled = true; };    // FP32, rolled, 85 regs
template <> struct TickBounds<10> { static constexpr int kThreads = 256, kMinBlocks = 1; static constexpr bool kRolled = false; };  // FP64
template <> struct TickBounds<kCoopVariant> { static constexpr int kThreads = 256, kMinBlocks = 1; static constexpr bool kRolled = false; };  // FP64, eight lanes per link

template <> struct TickBounds<kLanesVariant> { static constexpr int kThreads = 256, kMinBlocks = 1; static constexpr bool kRolled = false; };  // FP32, eight lanes per link
// FP32, one thread per link, begun before the previous launch has ended
// (k_update): all registers (at most 8 warps per SM), unrolled for 4-D tori
// and rolled.
constexpr int kEarlyVariant = 13, kEarlyRolled = 14;
template <int V>
constexpr bool kIsEarly = V == kEarlyVariant || V == kEarlyRolled;
// FP32, draws parked in shared memory: variants 0 and 1 otherwise.
constexpr int kParked0 = 15, kParked1 = 16;
template <int V>
constexpr bool kIsParked = V == kParked0 || V == kParked1;
// FP64, fused launches with two-coupling chains among others.
constexpr int kMixedVariant = 17;
template <> struct TickBounds<kMixedVariant> { static constexpr int kThreads = 256, kMinBlocks = 1; static constexpr bool kRolled = false; };
template <> struct TickBounds<kParked0> { static constexpr int kThreads = 256, kMinBlocks = 2; static constexpr bool kRolled = false; };
template <> struct TickBounds<kParked1> { static constexpr int kThreads = kParkedThreads1, kMinBlocks = 5; static constexpr bool kRolled = false; };
template <> struct TickBounds<kEarlyVariant> { static constexpr int kThreads = 256, kMinBlocks = 1; static constexpr bool kRolled = false; };
template <> struct TickBounds<kEarlyRolled> { static constexpr int kThreads = 256, kMinBlocks = 1; static constexpr bool kRolled = true; };

// ------------------------------------------------------------------ one tile of an update phase

// Book a warp's change of Re Tr(U A): each warp owns the slot of its links, so
// the one fire-and-forget add per warp meets no other add in this launch and
// the order of adds is fixed.
__device__ __forceinline__ void book_action(const ChainDesc &d, int slot, double sum) {
  if ((threadIdx.x & 31) == 0 && d.action_slots && in_bounds(slot, d.n_action_slots, kBoundsSlot))
    atomicAdd(d.action_slots + slot, d.action_factor * sum);
}
__device__ __forceinline__ double warp_sum(ActionChange dr) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dr.v += __shfl_down_sync(0xffffffffu, (long long)dr.v, o);
  double sum = dbl_of(dr.v, 51);
  if (__any_sync(0xffffffffu, dr.general != 0.0)) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dr.general += __shfl_down_sync(0xffffffffu, dr.general, o);
    sum += dr.general;
  }
  return sum;
}

// The links j0.. of one warp with eight lanes per link, in two parts: what
// needs no link (the site, the draws), and the update.
template <class S, bool SUB>
struct WarpLinks {
  using Draws = std::conditional_t<sizeof(typename S::R) == 8, CoopDraws, DrawPre>;
  SiteGeo g;
  int jj;
  bool valid;
  uint32_t c0;
  Draws draws;

  __device__ __forceinline__ void prepare(const ChainDesc &d, uint32_t sweep, int colour, int mu, int layer, int j0) {
    const int j = j0 + (int)(threadIdx.x & 31) / kCoopLanes;
    valid = j < d.Vn;
    jj = min(j, d.Vn - 1);
    g = site_of<SUB>(d, layer, colour, jj);
    c0 = site_key<SUB>(d, g);
    const uint2 key = make_uint2(d.seed_lo, d.seed_hi);
    if constexpr (sizeof(typename S::R) == 8)
      draws = coop_draws(key, c0, sweep, colour, mu);
    else
      draws = lanes_draws_f(key, c0, sweep, colour, mu);
  }

  // slot: the warp's action slot
  template <bool COH>
  __device__ __forceinline__ void update(const ChainDesc &d, uint32_t sweep, int colour, int mu, int slot,
                                         uint32_t &np, uint32_t &na) {
    if constexpr (sizeof(typename S::R) == 8) {
      ActionChange dr = {0, 0.0};
      update_site_coop<SUB, COH>(d, sweep, colour, mu, g, jj, c0, valid, draws, np, na, dr);
      __syncwarp();
      book_action(d, slot, warp_sum(dr));
    } else {
      float dr = 0.0f;
      update_site_lanes<S, SUB>(d, sweep, colour, mu, g, c0, valid, draws, np, na, dr);
      __syncwarp();
#pragma unroll
      for (int o = 16; o >= kCoopLanes; o >>= 1) dr += __shfl_down_sync(0xffffffffu, dr, o);
      book_action(d, slot, (double)dr);
    }
  }
};

// The lanes of a link and the first link of this warp in tile lt (slot: the
// warp's action slot).
template <int V>
constexpr int kLanesOf = V == kCoopVariant || V == kLanesVariant ? kCoopLanes : 1;
struct WarpPlace {
  int layer, jw, slot;
};
template <int LANES>
__device__ __forceinline__ WarpPlace warp_place(const ChainDesc &d, int lt) {
  constexpr int kPerWarp = 32 / LANES;
  WarpPlace p;
  p.layer = fast_div(lt, d.tdiv);  // a layer, or a sublattice box of one
  p.jw = (lt - p.layer * d.tiles_per_vl) * ((int)blockDim.x / LANES) + (int)(threadIdx.x & ~31u) / LANES;
  p.slot = p.layer * ((d.Vn + kPerWarp - 1) / kPerWarp) + p.jw / kPerWarp;
  return p;
}

// The updates of one CTA's tile lt of a chain's phase (colour, mu).
template <class S, int V, bool WT, bool SUB, bool TOR, class Ready = NotEarly>
__device__ __forceinline__ void update_tile(const ChainDesc &d, uint32_t sweep, int colour, int mu, int lt,
                                            uint32_t &np, uint32_t &na, Ready &&ready = Ready()) {
  const WarpPlace p = warp_place<kLanesOf<V>>(d, lt);
  const int layer = p.layer;
  if constexpr (kLanesOf<V> > 1) {
    if (p.jw >= d.Vn) return;
    WarpLinks<S, SUB> w;
    w.prepare(d, sweep, colour, mu, layer, p.jw);
    w.template update<false>(d, sweep, colour, mu, p.slot, np, na);
  } else {
    const int jj = p.jw + (int)(threadIdx.x & 31);
    const bool valid = jj < d.Vn;
    double sum = 0.0;
    // the one-coupling FP64 update runs in fixed point, also beside chains of
    // two couplings: a chain's links do not depend on the others of its launch
    constexpr bool kMixed = V == kMixedVariant;
    constexpr bool kFixed = std::is_same<S, StoreF64x18>::value && (!WT || kMixed);
    if (kFixed && !(kMixed && d.weighted)) {
      if constexpr (kFixed) {
        ActionChange dr = {0, 0.0};
        if (valid) update_site_fixed<SUB>(d, sweep, colour, mu, layer, jj, np, na, dr);
        __syncwarp();
        sum = warp_sum(dr);
      }
    } else if constexpr (!kFixed || kMixed) {
      typename S::R dr = 0;  // in the kernel's precision
      if (valid) {
        if constexpr (kIsEarly<V> && TickBounds<V>::kRolled)
          update_site<S, true, WT, SUB, true>(d, sweep, colour, mu, layer, jj, np, na, dr, ready);
        else if constexpr (kIsEarly<V>)
          update_site_lean<S, false, 4, 1>(d, sweep, colour, mu, layer, jj, np, na, dr, ready);
        else if constexpr (kIsParked<V>)
          update_site_lean<S, false, TOR ? 4 : 0, 2>(d, sweep, colour, mu, layer, jj, np, na, dr, ready);
        else if constexpr (TOR)
          update_site_lean<S, false, 4>(d, sweep, colour, mu, layer, jj, np, na, dr);
        else if constexpr (!TickBounds<V>::kRolled && !SUB)
          update_site_lean<S, WT>(d, sweep, colour, mu, layer, jj, np, na, dr);
        else
          update_site<S, TickBounds<V>::kRolled, WT, SUB>(d, sweep, colour, mu, layer, jj, np, na, dr);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dr += __shfl_down_sync(0xffffffffu, dr, o);
      sum = (double)dr;
    }
    // (a warp of the ragged last tile with no link has no slot)
    if (p.jw < d.Vn) book_action(d, p.slot, sum);
  }
}

// ------------------------------------------------------------------ launching

// Every kernel may be scheduled before the previous one of the stream has
// finished (programmatic launch): wait for its completion and memory before
// touching anything, then let the next kernel be scheduled.  Both are no-ops
// for an ordinary launch.
__device__ __forceinline__ void wait_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// pdl: launch as a programmatic dependent of the previous kernel in the
// stream (the kernel waits for that one's completion and memory at its first
// instruction, so only the launch itself overlaps the previous kernel).
template <class... P, class... A>
static cudaError_t launch_shared(void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, bool pdl,
                                 A &&...a) {
  cudaLaunchConfig_t cfg = {};
  cfg.dynamicSmemBytes = smem;
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)block);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(a)...);
}
template <class... P, class... A>
static cudaError_t launch_ex(void (*kernel)(P...), dim3 grid, int block, cudaStream_t st, bool pdl, A &&...a) {
  return launch_shared(kernel, grid, block, 0, st, pdl, std::forward<A>(a)...);
}

// Run f with a value of the storage form of `storage` (0: FP64 18-real,
// 1: FP32 12-real, 2: FP32 18-real); f launches the kernels of that form.
template <class F>
static inline cudaError_t by_storage(int storage, F &&f) {
  switch (storage) {
    case 0: return f(StoreF64x18{});
    case 2: return f(StoreF32x18{});
    default: return f(StoreF32x12{});
  }
}

}  // namespace su3g
