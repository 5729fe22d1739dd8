// su3_engine.h -- data structures shared by the host runtime and the kernels.
//
// The engine advances a set of resident chains (lattices).  Each launch of
// the tick kernel moves every active chain one stage forward: one
// (colour, direction) phase of the checkerboard sweep, or a
// re-unitarisation, or a measurement.  The stage machine lives in device
// memory, so a captured graph of ticks replays without host involvement and
// chains of different D can share a launch.  Every chain has two state
// slots, and a launch reads slot `parity`.  With several chains, the first
// warp of a launch to finish writes every chain's next state into the other
// slot while the rest of the launch runs, and the last one finishes the
// tick's measurements and flips the parity; a single chain is advanced in
// place by the launch's last warp.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace su3g {

constexpr int kMaxD = 4;

// Stages beyond the 2D update phases.
constexpr int kStageReunit = 100;
constexpr int kStageMeasure = 101;

// Random-number stream purposes (fourth Philox counter word).
constexpr uint32_t kPurposeHeatbath = 0u;
constexpr uint32_t kPurposeStart = 1u;
constexpr uint32_t kHitDirection = 255u;

// FP32 storage: an SU(2) draw with alpha at or above this value is taken in
// double precision from the full 32-bit random words (weak-coupling links,
// where X ~ 1/alpha is small and its relative precision sets the size of
// the rotation).
constexpr float kAlphaFp64 = 32.0f;
// FP32 storage: below this alpha (strong coupling) the float draw takes the
// accurate logf / cosf instead of their SFU forms (their absolute errors
// would be divided by alpha).
constexpr float kAlphaAccurateLog = 2.0f;

// FP64 chains of one coupling with at most kCoopSites links per update phase
// take eight lanes per link (update_site_coop): a tile then holds an eighth
// of a CTA's threads.  In 4-D one thread per link takes 33 us per phase for
// any lattice below one wave (38912 links at 8 warps per SM), eight lanes 12
// us for few links, 16 for a full wave of 4864 and 30.4 for 8192 links.  A
// one-chain engine of fewer dimensions has fewer staples than lanes and leaves
// them sooner.  With and without lanes, 3-D: 22^3 (5324 links) 26.2 and 27.3
// us, 24^2 x 22 (6336) 28.9 and 27.3, 24^3 (6912) 30.1 and 27.7; 2-D: 96 x 100
// (4800) 17.0 and 21.0, 108 x 100 (5400) 27.7 and 22.3, 128^2 32.7 and 22.0.
constexpr int kCoopLanes = 8;
constexpr int kCoopSites = 8192, kCoopSites3 = 5632, kCoopSites2 = 4864;

// Float chains of one coupling with at most kLanesLinks links per phase take
// eight lanes per link too (update_site_lanes; the launchers' variant
// kFloatLanes): one warp per scheduler.  Per phase, against one thread per
// link (kFloatEarly below): 12^2 x 8 x 4 (2304 links) 4.05 us and 4.20, 8^4 in
// four boxes 4.6 and 5.6; 12^3 x 4 (3456) 4.68 and 4.16, 16^2 x 8 x 4 (4096)
// 5.7 and 4.2.
constexpr int kLanesLinks = 2432, kFloatLanes = 16;
// The launchers' variants of the float updates that begin before the previous
// launch has ended, one thread per link: the second is rolled, and the first
// too unless the chain is an undivided 4-D torus with the default keys.
constexpr int kFloatEarly = 17, kFloatEarlyRolled = 18;
// The launchers' variants of the float updates whose draws alone come before
// that wait (128 and 96 registers; the second up to kParkedThreads1 threads).
constexpr int kFloatParked0 = 19, kFloatParked1 = 20, kParkedThreads1 = 128;
// Chains of one coupling with at most kClusterLinks links per phase run whole
// sweeps in one launch of a cluster of CTAs (k_sweeps), eight lanes per link.
// Per phase, against a launch per phase: float 4^4 3.25 us (3.62), 8^3 3.22
// (3.77), 16^2 3.78 (4.57); FP64 4^4 11.4 (11.6), 8^3 11.6 (12.1).  More links
// share the cluster's 16 SMs too long: float 8^3 x 4 6.3 us against 4.3, both
// with the draws after the wait.
constexpr int kClusterCtas = 16, kClusterThreads = 128;
constexpr int kClusterLinks = kClusterCtas * kClusterThreads / kCoopLanes;

// Pairs of FHKP counters per chain (their sums are the totals).
constexpr int kCounterSlots = 32;
// A measurement's partial sums: at most this many CTAs per layer (one wave: 5
// per SM, FP64 3).
constexpr int kMeasureCtas = 760, kMeasureCtasF64 = 456;
// Float measurements of at most this many sites per colour take eight lanes
// per site.
constexpr int kSplitSites = 4096;

// Results per measurement slot: [total, space, time, poly_re, poly_im].
constexpr int kMeasVals = 5;
// Partial sums per tile in a measurement: [space, time, poly_re, poly_im].
constexpr int kPartVals = 4;

// Division of 0 <= r < 2^31 by a number fixed on the host: (hi(m r) + r) >> s
// (Granlund and Montgomery; three instructions instead of about twenty).
struct FastDiv {
  uint32_t m, s;
};
inline FastDiv fast_div_of(uint32_t n) {
  uint32_t s = 0;
  while (s < 31 && (1u << s) < n) ++s;
  return {(uint32_t)((((1ull << s) - n) << 32) / n + 1), s};
}

struct ChainDesc {
  void *links;               // storage base (Vec units, see su3_device.cuh)
  double *results;           // [result_cap][nlayers + 1][kMeasVals]
  double *partials;          // [tiles][kPartVals]
  unsigned long long *counters;  // [kCounterSlots][proposals, accepts]
  double *action_slots;      // booked action changes, one slot per warp of sites: [layer][ceil(Vh/32)]
  double *ref_meas;          // the measurement the booked changes count from: [nlayers + 1][kMeasVals]
  int32_t n_action_slots;
  uint32_t seed_lo, seed_hi;
  int32_t D, nlayers, glue_mask, layer_blind;
  int32_t custom_period;     // 0: site key = layer*V + i_s - 1
  int32_t dims[kMaxD];
  int32_t period[kMaxD];
  int32_t stride[kMaxD];     // n_a^i of eq. (i_s)
  int32_t pstride[kMaxD];    // strides of the random-number period lattice
  int32_t V, Vh, Vp;         // sites per layer, per colour and layer, per period lattice
  int32_t hits;
  int32_t reunit_every, measure_every;
  int32_t tiles_per_layer;   // ceil(Vh / tile)
  int32_t tile_base;         // first global tile of this chain
  int32_t result_cap;
  int32_t spatial_per_layer; // V / n^D (Polyakov lines per layer)
  int32_t pow2;              // 1: every extent is a power of two (coordinates by shifts)
  int32_t shift[kMaxD];      // log2 n^i when pow2
  // Sublattice decomposition on one device (the paper's MPI sublattices,
  // Sec. 2.4): nb sublattices per layer, each stored as its own padded box
  // (interior idims plus one halo layer on both sides where hpad = 1), the
  // boxes side by side as virtual layers vl = layer * nb + block.  In that
  // case dims / stride / Vh describe the padded box, V the undivided layer
  // and gstride its strides (random-number site key).  Undivided: nb = 1,
  // idims = dims, hpad = 0, bdiv = 1, Vn = Vh.
  int32_t nb;
  int32_t tiles_per_vl;      // ceil(Vn / tile); tiles_per_layer = nb * tiles_per_vl
  int32_t Vn;                // sites of one colour updated per virtual layer
  int32_t idims[kMaxD];      // interior extents
  int32_t hpad[kMaxD];       // 1: divided direction, one halo layer on each side
  int32_t bdiv[kMaxD];       // sublattices per direction
  int32_t gstride[kMaxD];    // strides of the undivided layer
  FastDiv idiv[kMaxD], bdivf[kMaxD];  // division by idims, bdiv
  FastDiv tdiv;              // division by tiles_per_vl
  // Halo sites of a box (the same for every box), colour 0 first then
  // colour 1: {padded index, owner's padded index, owner box offset code
  // (2 bits per direction: 0 same box, 1 previous, 2 next), 0}.
  const int4 *halo;
  int32_t halo_n[2];
  float beta_f;
  double beta_d;
  // DLT with two couplings (Sec. 2.2): weighted = 1 when beta1 != beta; a
  // plaquette with any link in layer 1 then has beta1, and the staple is
  // accumulated with these weights (the heatbath runs with beta = 1).
  int32_t weighted;
  float beta1_f;
  double beta1_d;
  // 3 / (2 beta) = inv_beta_m 2^-60 2^inv_beta_e, the mantissa in [1/2, 1)
  // (beta = 0: an exponent beyond any acceptance): the fixed-point draw
  int64_t inv_beta_m;
  int32_t inv_beta_e;
  double action_factor;      // booked dS per unit change of Re Tr(U A): -beta/3, or -1/3 when weighted
};

struct ChainState {
  uint32_t sweep;          // completed sweeps (the random-number sweep counter)
  int32_t stage;           // 0..2D-1: update phase colour*D + mu; kStageReunit; kStageMeasure
  uint32_t target;         // the chain goes idle at the start of this sweep
  int32_t active;          // 1: advancing; 0: idle
  uint32_t n_meas;         // measurements recorded
  int32_t anchor;          // 1: the next measurement restarts the action bookkeeping
  int32_t pad[2];
};

// The device side of a one-chain engine's fixed schedule.  The sweep counter
// has two copies: the launches of one graph read `cur` (its first launch
// copies `nxt` there), and its last launch writes `nxt`, so that no launch
// reads a word that its own CTAs write.
struct ChainCtl {
  uint32_t cur, nxt;
  uint32_t n_meas;         // measurements recorded
  int32_t anchor;          // 1: the next measurement restarts the action bookkeeping
  uint32_t done;           // CTAs of a measurement that have written their partial sums
  int32_t pad[3];
};

// One update phase of a fixed schedule.
struct UpdateStep {
  int32_t colour, mu;
  uint32_t offset;         // sweeps completed since the schedule's first launch
  uint32_t advance;        // last launch: sweeps to add to the counter (0: not the last)
  int32_t first;           // 1: the schedule's first launch
  int32_t early;           // 1: its third or a later one: `cur` may be read before the previous launch has ended
  int32_t tiles;
};

struct EngineHeader {
  int32_t nchains;
  int32_t total_tiles;
  int32_t tile;            // threads per CTA = sites per tile
  int32_t parity;          // the state slot that holds every chain's current state
  uint32_t done;           // warps counted (bits 0-30); bit 31: some chain measures in this tick
  int32_t n_meas;          // chains entered in meas_list by this launch
  int32_t pad[2];
};

struct EngineArgs {
  ChainDesc *desc;
  ChainState *state;       // [chain][2]: slot parity current, the other one next
  EngineHeader *hdr;
  int32_t *tile_chain;     // [total_tiles] -> chain
  int32_t *meas_list;      // [chains] chains whose measurement the last warp finishes
};

}  // namespace su3g
