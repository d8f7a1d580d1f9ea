// Host-side launch interface between the C-ABI layer and the kernels.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "tracer.cuh"

namespace mcbte {

// Per-geometry inputs of the setup kernel, passed by value (4 KB): the
// descriptor, the particles of this call, the index of the first one, and
// the particles of the whole run that normalise E_eff = E_tot / N.
struct SetupArgs {
  const mcbte_geometry_desc* desc[kMaxGeoms];
  uint64_t n[kMaxGeoms];
  uint64_t pid0[kMaxGeoms];
  uint64_t n_norm[kMaxGeoms];
  int cut_flights;   // no flight runs through periodic faces (GeoRun::unfold stays 0)
};

int sm_count();

// FP64 tracers: one block of six warps per SM, or fewer blocks where the run
// has no particles for them.  An FP64 warp instruction takes 64 cycles of its
// scheduler's pipe, one warp nearly fills it, and every further warp makes the
// longest particle's events wait (silicon-like slab, 3e5 particles, up to 2100
// events each: 21.9 ms at 16 warps a SM, 17.2 at 8, 16.0 at 6, 15.2 at 4; 2e6
// particles: 58.9, 54.2, 54.4, 63.0).
constexpr int kF64Threads = 192;
constexpr int kF64RegionThreads = 128;   // k_transient_fp64_regions: one warp per scheduler
inline int f64_blocks(uint64_t total) {
  const uint64_t most = (uint64_t)sm_count();   // a warp on every SM first
  return (int)(total < most ? total : most);
}

cudaError_t launch_setup(const SetupArgs& a, int n_geoms, const MatView& M, int transient, double t_max_s,
                         int tally_axis, GeoRun* geos, uint64_t* offs, unsigned long long* t0, cudaStream_t s);

cudaError_t launch_steady(int precision, bool grad, const GeoRun* geos, const uint64_t* offs, const MatView& M,
                          const RunCfg& C, const Acc& A, int threads, int blocks_per_sm, cudaStream_t s);

struct SteadyOutDev {
  double* T;
  double* q;
  double* q_bin;
  double* stats;
  double* dk;        // grad: [n_bins]
  double* dkp;       // grad: [2]
  double* dkdir;     // grad: [n_dirs][2]
  double* det;       // detector regions: [n_det][4], or null
  double* kn;        // N_scat_max curve: [G][n_scat_max][2], or null
};

cudaError_t launch_steady_f32(bool grad, bool cells, const GeoRun* geos, const uint64_t* offs, const MatView& M,
                              const RunCfg& C, const Acc& A, int threads, int bps, cudaStream_t s);
// the same with the main kernel that parks its tail and the tail kernel
cudaError_t launch_steady_f32_tail(bool grad, bool cells, const GeoRun* geos, const uint64_t* offs, const MatView& M,
                                   const RunCfg& C, const Acc& A, int threads, int bps, cudaStream_t s);
cudaError_t launch_transient_f32(const GeoRun* geos, const MatView& M, const RunCfg& C, const Acc& A, int threads,
                                 int bps, cudaStream_t s);

cudaError_t launch_finalize_steady(const GeoRun* geos, const MatView& M, const RunCfg& C, const Acc& A,
                                   const SteadyOutDev& O, bool grad, const int* flags, cudaStream_t s);

cudaError_t launch_dirs_dot_pi(const double* dirs, int n_dirs, const MatView& M, double* dpi, cudaStream_t s);

cudaError_t launch_transient(int precision, const GeoRun* geos, const MatView& M, const RunCfg& C, const Acc& A,
                             int threads, int blocks_per_sm, cudaStream_t s);

cudaError_t launch_finalize_transient(const GeoRun* geos, const MatView& M, const RunCfg& C, const Acc& A,
                                      double* tally, double* stats, size_t n_cells_total, bool fixed,
                                      cudaStream_t s);

// Material table build (FP64): per-bin kernel + one block per alias table.
struct MatBuild {
  int n;
  const double *omega, *v, *tau, *C_in, *D, *domega;
  const double* tau_imp;   // optional two-phonon relaxation times (s), or null
  const double* spec_bin;  // optional per-bin specularity, or null
  uint64_t* spec_thr;      // [n] its thresholds (when given)
  double T_lin;
  double *C, *w_emit, *w_init, *w_relax, *v_nm, *inv_v, *lam, *pi, *sums;
  double* lam2;            // [n] v tau_imp (nm), +inf without a two-phonon clock
  double* prob;        // [3][n]
  uint64_t* thr;       // [3][n]
  int32_t* alias;      // [3][n]
  uint4* rec;          // [3][n]
  float4* binf;        // [n]
  double* scratch_p;   // [3][n]
  int* scratch_small;  // [3][n]
  int* scratch_large;  // [3][n]
};

cudaError_t launch_material_build(const MatBuild& b, cudaStream_t s);

// Particle indices a warp takes at once: a multiple of 32, at most `most` (one
// returning atomic per chunk), and about four chunks per warp of the grid, so
// that a run of few particles spreads over all of them.  Runs of 256 left 16 warps of 3648 with
// work at 4096 particles and 391 at 100 000 (gray slab of 1e5 particles: main
// kernel 212 us, 35 us with runs of 32 and the block's sums in BlockAcct).
inline unsigned take_chunk(uint64_t total, uint64_t warps, unsigned most) {
  const uint64_t c = (total / (4 * warps)) & ~(uint64_t)31;
  return c < 32 ? 32u : (c > most ? most : (unsigned)c);
}
// The same where the particles fit the lanes of `spread` warps: an equal share
// each (at least `least`) and no counter.  The fewer lanes a warp carries, the
// fewer branches its events take one after the other.  FP64: one warp per
// scheduler, whose pipe it fills (pore film, 2000 particles 1.80 -> 1.62 ms;
// hot spot, 5000 2.01 -> 1.65; beyond 32 x 4 warps per SM 20 000 particles take
// 8.65 ms either way).  FP32: all warps, 4 lanes at least, also where the warps
// park what they hold at once (us with shares of 16, 8 and 4: gray slab of 4096
// particles 116, 108, 109; silicon-like slab of 4096 1422, 1200, 1199; pore
// film of 2000 183, 170, 170; 20 films of 100 each 201, 154, 152).
inline unsigned take_chunk(uint64_t total, uint64_t warps, unsigned most, uint64_t spread, unsigned least) {
  if (total > 32 * spread) return take_chunk(total, warps, most);
  const uint64_t c = (total + spread - 1) / spread;
  return c < least ? least : (unsigned)c;
}

// bytes of one parked particle of the FP32 steady tracer's tail (both passes)
size_t park_record_bytes();

}  // namespace mcbte
