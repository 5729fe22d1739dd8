// su3_launch.h -- host-side entry points of the kernels.
#pragma once
#include <cuda_runtime.h>

#include "su3_engine.h"

namespace su3g {

// storage: 0 = FP64 18-real, 1 = FP32 12-real, 2 = FP32 18-real.
// The update comes in variants (FP32 12-real: 0 = 128, 1 = 96 registers;
// 2 = 96, 3 = 128, 4 = 85 registers with a rolled staple loop; FP32 18-real:
// 0; FP64: 0, and 1 = eight lanes per link); a variant limits the CTA width to
// tick_max_threads.  weighted selects the form compiled for two-coupling DLT
// chains (needed when any chain of the launch has beta1 != beta); torus the
// form for undivided periodic 4-D tori with one coupling and the default
// random-number key (ignored where none exists).
int tick_variants(int storage);
int tick_max_threads(int storage, int variant);
// One tick of many chains: each at its own stage.
cudaError_t launch_tick(int storage, int variant, bool weighted, bool torus, const EngineArgs &ea, int grid, int block,
                        cudaStream_t st, bool pdl);
cudaError_t tick_occupancy(int storage, int variant, bool weighted, bool torus, int block, int *ctas_per_sm);

// One chain: an update phase, a re-unitarisation, a measurement (into out, or
// recorded in the chain's ring and ctl).  sub: the chain is divided into
// sublattice boxes (it fixes the FP32 variant: 3).
cudaError_t launch_update(int storage, int variant, bool weighted, bool sub, bool torus, const ChainDesc &d,
                          ChainCtl *ctl, const UpdateStep &step, int grid, int block, cudaStream_t st, bool pdl);
cudaError_t update_occupancy(int storage, int variant, bool weighted, bool sub, bool torus, int block,
                             int *ctas_per_sm);
// Whole sweeps of a small one-coupling chain in one launch (at most
// kClusterLinks links per phase).
bool sweeps_supported(int storage, bool sub);
cudaError_t launch_sweeps(int storage, bool sub, const ChainDesc &d, ChainCtl *ctl, int sweeps, cudaStream_t st,
                          bool pdl);
// The same of FP64 chains (su3_update64.cu), to which the above pass them.
cudaError_t launch_update64(int variant, bool weighted, bool sub, const ChainDesc &d, ChainCtl *ctl,
                            const UpdateStep &step, int grid, int block, cudaStream_t st, bool pdl);
cudaError_t update_occupancy64(int variant, bool weighted, bool sub, int block, int *ctas_per_sm);
bool sweeps_supported64(bool sub);
cudaError_t launch_sweeps64(bool sub, const ChainDesc &d, ChainCtl *ctl, int sweeps, cudaStream_t st, bool pdl);

cudaError_t launch_reunit(int storage, bool sub, const ChainDesc &d, cudaStream_t st, bool pdl);
cudaError_t launch_measure(int storage, bool sub, const ChainDesc &d, double *out, ChainCtl *ctl, cudaStream_t st,
                           bool pdl);
cudaError_t launch_set_ctl(ChainCtl *ctl, uint32_t sweep, uint32_t n_meas, int anchor, cudaStream_t st);

// Refresh every halo of a divided chain (after a start, new links or a
// re-unitarisation; update phases write the copies of their links
// themselves), and the copies between its sublattice boxes and the undivided
// layout.  halo_sites: halo sites of one box (both colours).
cudaError_t launch_halo(int storage, const ChainDesc &d, int halo_sites, cudaStream_t st, bool pdl = false);
cudaError_t launch_sub_copy(int storage, const ChainDesc *sub_dev, const ChainDesc *plain_dev, size_t nlinks,
                            int to_sub, cudaStream_t st);
cudaError_t launch_start(int storage, const ChainDesc &d, size_t nlinks, int hot, cudaStream_t st);
cudaError_t launch_convert(int storage, const ChainDesc &d, size_t nlinks, double *canon, int to_canonical,
                           cudaStream_t st);
// Links from rows 1, 2 in float (12 per link, canonical order; 16-byte aligned).
cudaError_t launch_convert_rows2(int storage, const ChainDesc &d, size_t nlinks, const float *src, cudaStream_t st);
void host_advance_stage(const ChainDesc &d, ChainState &s);
// Fixed-order sum of n booked action-change slots into *out (device).
cudaError_t launch_action_sum(const double *slots, int n, double *out, cudaStream_t st);
cudaError_t launch_arm(ChainState *state, int nchains, uint32_t n, cudaStream_t st);
cudaError_t launch_set_anchor(ChainState *state, int value, cudaStream_t st);
// Measurement with partial sums in the library's static device scratch
// (su3_measure_noalloc); the descriptor is passed by value.
int noalloc_max_tiles();
// Debug-bounds builds (SU3_DEBUG_BOUNDS): whether this is one, the first
// recorded violation (site, index, extent; site 0: none), and a self-test
// that records a deliberate violation without any memory access.
bool debug_bounds_build();
cudaError_t bounds_record(unsigned long long out[3]);  // of su3_kernels.cu, then of the other units
cudaError_t bounds_record_tick(unsigned long long out[3]);
cudaError_t bounds_record_update(unsigned long long out[3]);
cudaError_t bounds_record_update64(unsigned long long out[3]);
cudaError_t bounds_record_stages(unsigned long long out[3]);
cudaError_t launch_bounds_selftest();
cudaError_t launch_measure_noalloc(int storage, const ChainDesc &d, int block, double *out, cudaStream_t st);

}  // namespace su3g
