// Steady-state tracing (Sec. 3.6, Eq. steady_estimate): the persistent FP64
// plain kernel (FP64 throughout) and the persistent FP32 kernel (FP32 flights;
// 64-bit fixed-point tallies privatised in shared memory, reduced to FP64;
// alias tables in shared memory), plus the finalisation kernel.  In both a lane
// that is done takes its warp's next particle, from the run of indices that the
// warp holds or takes from the work counter (WarpRun).
//
// This file is compiled three times: with MCBTE_F64 (FP64 kernels, no fused
// multiply-add) and with MCBTE_F32 twice, MCBTE_F32_PART 0 (the FP32 kernels
// of runs without the tail kernel, and the launch dispatch) and 1 (the FP32
// kernels that park their tail, and the tail kernels), built in parallel.
#include <atomic>

#include "launch.h"
#include "tail.cuh"

#ifndef MCBTE_F64
#define MCBTE_F64 0
#endif
#ifndef MCBTE_F32
#define MCBTE_F32 0
#endif
#ifndef MCBTE_F32_PART
#define MCBTE_F32_PART 0
#endif

namespace mcbte {

namespace {

// N_scat_max curve: a trajectory that ended (absorbed, truncated) after m <
// n_scat_max relaxations has the same final tally X in every run with
// N_scat_max > m; it enters the difference array at m + 1.
__device__ __forceinline__ void nscat_end(const RunCfg& C, int g, int m, double X) {
  if (!C.nscat_acc || m >= C.n_scat_max) return;
  double* a = nscat_slot(C, g, m + 1);
  atomicAdd(a + 2, X);
  atomicAdd(a + 3, X * X);
}

// Likelihood-ratio contributions of a finished particle with tally X: every
// relaxation period's value into G[bin], the dense resampling term R, the
// specularity score and the probe directions.
template <class Grad>
__device__ __forceinline__ void grad_finish(const Grad& gr, double X, int g, const RunCfg& C, const Acc& A,
                                            const MatView& M) {
  const int np = gr.periods();
  for (int k = 0; k < np; ++k) atomicAdd(&A.G[gr.period_bin(k)], gr.period_value(k, X));
  const double Rv = gr.resample_term(X);
  double* gs = grad_copy(A);
  atomicAdd(gs + 0, Rv);
  if (!C.mvd) {   // the measure-valued score is added after the phantom trace
    const double gp = gr.spec_term(X);
    atomicAdd(gs + 1, gp);
    atomicAdd(gs + 2, gp * gp);
  }
  for (int kd = 0; kd < C.n_dirs; ++kd) {
    const double* dd = C.dirs + (size_t)kd * M.n;
    double val = 0.0;
    for (int k = 0; k < np; ++k) val += gr.period_value(k, X) * dd[gr.period_bin(k)];
    val += Rv * C.dpi[kd];
    atomicAdd(gs + 4 + 2 * kd, val);
    atomicAdd(gs + 5 + 2 * kd, val * val);
  }
}

template <bool GRAD, class On>
struct GradPick { using type = On; };
template <class On>
struct GradPick<false, On> { using type = GradOff; };

// Per-thread book-keeping of finished particles (integer / fixed-point
// fields, few registers), flushed to the geometry's global accumulators when
// the thread moves to another geometry and at exit.
// SX: the tally's type, 2^-20 nm whole numbers (FP32 path, exact) or FP64 nm.
__device__ __forceinline__ double tally_nm(long long x) { return (double)x * kFxInv; }
__device__ __forceinline__ double tally_nm(double x) { return x; }

template <typename SX>
struct ThreadAcct {
  int g;
  unsigned traced, trunc, absorbed, maxev;
  int s_emit, s_abs;
  unsigned long long ev;
  SX sx;              // sum of X
  double sx2;

  __device__ __forceinline__ void reset(int gg) {
    g = gg;
    traced = trunc = absorbed = maxev = 0u;
    s_emit = s_abs = 0;
    ev = 0ull;
    sx = SX(0);
    sx2 = 0.0;
  }
  // a particle with tally X (x in the tally's type) ended with `out` after nev events
  __device__ __forceinline__ void end(int out, unsigned nev, int sgn, SX x, double X) {
    ev += nev;
    trunc += (out == STEP_TRUNCATED) ? 1u : 0u;
    maxev = nev > maxev ? nev : maxev;
    traced += 1u;
    sx += x;
    sx2 += X * X;
    s_emit += sgn;
    if (out == STEP_ABSORBED) {
      s_abs += sgn;
      absorbed += 1u;
    }
  }
  __device__ __forceinline__ void flush(const Acc& A) const {
    if (g < 0 || traced == 0u) return;
    atomicAdd(&A.cnt[g * 4 + 0], ev);
    if (trunc) atomicAdd(&A.cnt[g * 4 + 1], (unsigned long long)trunc);
    atomicMax(&A.cnt[g * 4 + 2], (unsigned long long)maxev);
    atomicAdd(&A.cnt[g * 4 + 3], (unsigned long long)traced);
    atomicAdd(&A.dsc[g * 8 + 0], tally_nm(sx));
    atomicAdd(&A.dsc[g * 8 + 1], sx2);
    atomicAdd(&A.dsc[g * 8 + 2], (double)s_emit);
    if (absorbed) {
      atomicAdd(&A.dsc[g * 8 + 3], (double)s_abs);
      atomicAdd(&A.dsc[g * 8 + 7], (double)absorbed);
    }
  }
};

// The sum of the block's tallies.  A lane's sum fits 64 bits (2^43 nm), a
// block's need not (gray, 30 m free path: 2e5 particles wrapped), so a block
// adds the halves apart, the upper one signed; whole numbers, hence the same
// sum in any order.
template <typename SX> struct BlockSum;
template <> struct BlockSum<long long> {
  long long hi, lo;
  __device__ __forceinline__ void reset() { hi = lo = 0; }
  // x: this lane's; called by all 32 lanes, lane 0 adds
  __device__ __forceinline__ void add(long long x) {
    long long h = x >> 32, l = (long long)(unsigned)x;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      h += __shfl_xor_sync(0xffffffffu, h, o);
      l += __shfl_xor_sync(0xffffffffu, l, o);
    }
    if ((threadIdx.x & 31u) != 0u) return;
    red_s64(&hi, h);
    red_s64(&lo, l);
  }
  __device__ __forceinline__ double nm() const { return ((double)hi * 4294967296.0 + (double)lo) * kFxInv; }
};
template <> struct BlockSum<double> {
  double v;
  __device__ __forceinline__ void reset() { v = 0.0; }
  __device__ __forceinline__ void add(double x) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31u) == 0u) atomicAdd(&v, x);
  }
  __device__ __forceinline__ double nm() const { return v; }
};

// A block's book-keeping (shared memory), for runs of one geometry.  Every
// lane of the grid flushing its own fields queued 8e5 atomics on seven
// addresses (about 0.4 ms, whatever the run's length: a gray slab of 1e5
// particles 502 us, 35 us without them); a warp's lanes are summed by
// shuffles, the block's warps here, and a block adds once.
template <typename SX>
struct BlockAcct {
  unsigned long long ev, trunc, maxev, traced;
  long long s_emit, s_abs, absorbed;
  BlockSum<SX> sx;
  double sx2;

  __device__ __forceinline__ void reset() {
    ev = trunc = maxev = traced = 0ull;
    s_emit = s_abs = absorbed = 0;
    sx.reset();
    sx2 = 0.0;
  }
  // called by all 32 lanes of a warp
  __device__ __forceinline__ void add(const ThreadAcct<SX>& t) {
    constexpr unsigned kAll = 0xffffffffu;
    unsigned long long ev_w = t.ev;
    long long se = t.s_emit, sa = t.s_abs;
    double s2 = t.sx2;
    unsigned long long tr = t.traced;
    const unsigned tc = __reduce_add_sync(kAll, t.trunc), ab = __reduce_add_sync(kAll, t.absorbed);
    const unsigned mx = __reduce_max_sync(kAll, t.maxev);
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      ev_w += __shfl_xor_sync(kAll, ev_w, o);
      se += __shfl_xor_sync(kAll, se, o);
      sa += __shfl_xor_sync(kAll, sa, o);
      s2 += __shfl_xor_sync(kAll, s2, o);
      tr += __shfl_xor_sync(kAll, tr, o);
    }
    if (tr == 0ull) return;   // the same in every lane
    sx.add(t.sx);
    if ((threadIdx.x & 31u) != 0u) return;
    atomicAdd(&ev, ev_w);
    if (tc) atomicAdd(&trunc, (unsigned long long)tc);
    atomicMax(&maxev, (unsigned long long)mx);
    atomicAdd(&traced, tr);
    atomicAdd(&sx2, s2);
    red_s64(&s_emit, se);
    if (ab) {
      red_s64(&s_abs, sa);
      red_s64(&absorbed, (long long)ab);
    }
  }
  // by one thread, after the block's warps have added
  __device__ __forceinline__ void flush(const Acc& A) const {
    if (traced == 0ull) return;
    atomicAdd(&A.cnt[0], ev);
    if (trunc) atomicAdd(&A.cnt[1], trunc);
    atomicMax(&A.cnt[2], maxev);
    atomicAdd(&A.cnt[3], traced);
    atomicAdd(&A.dsc[0], sx.nm());
    atomicAdd(&A.dsc[1], sx2);
    atomicAdd(&A.dsc[2], (double)s_emit);
    if (absorbed) {
      atomicAdd(&A.dsc[3], (double)s_abs);
      atomicAdd(&A.dsc[7], (double)absorbed);
    }
  }
};

#if MCBTE_F64
// ------------------------------------------------------------------ FP64 plain
// Persistent: a warp emits 32 particles at a time and a lane that is done
// takes the next one (Refill).  The FP64 pipe bounds the kernel, a warp
// instruction taking 64 cycles whether one lane or 32 are active; with a
// thread per particle 3.8 lanes were, most of them waiting for their warp's
// longest particle (silicon-like slab, 3e5 particles: 80.1 ms, now 16.0).
template <bool CELLS, bool GRAD>
__global__ void __launch_bounds__(kF64Threads, 1) k_steady_fp64(const GeoRun* __restrict__ geos,
                                                                const uint64_t* __restrict__ offs, MatView M, RunCfg C,
                                                                Acc A) {
  __shared__ Refill s_refill[kF64Threads / 32];
  __shared__ EmitBatch<double, true, false> s_batch[kF64Threads / 32];
  __shared__ BlockAcct<double> s_acct;
  if (threadIdx.x == 0) s_acct.reset();
  __syncthreads();
  constexpr unsigned kAll = 0xffffffffu;
  const unsigned lane = threadIdx.x & 31u;
  const uint64_t deadline = *C.t0 + C.budget_ns;
  const uint2 key = run_key(C);
  Refill& refill = s_refill[threadIdx.x >> 5];
  EmitBatch<double, true, false>& batch = s_batch[threadIdx.x >> 5];
  refill.start(lane, C.take_chunk, C.total, deadline, A.flags);
  Particle<double> p;
  using GradT = typename GradPick<GRAD, GradList>::type;
  GradT gr;
  if constexpr (GRAD) gr.mvd = C.mvd != 0;
  ThreadAcct<double> acct;
  acct.reset(-1);
  TallyPlain T;
  T.nc = C.n_cells;
  T.ca = C.cell_axis;
  T.ta = C.tally_axis;
  T.cP = T.qb = nullptr;
  T.h = 1.0;
  T.inv_h = 1.0f;
  T.det = nullptr;
  const size_t copy = blockIdx.x & (unsigned)(C.f64_rep - 1);   // of the cell and per-bin sums
  const GeoRun* G = geos;
  double X_nom = 0.0;   // gradient: the nominal trace's tally while the phantom runs
  bool alive = false, pool_dry = false;
  for (;;) {
    const unsigned need = __ballot_sync(kAll, !alive);
    if (need && !pool_dry) {
      pool_dry = refill.hand_out(
          32, need, lane, A.work, C.total, deadline, A.flags,
          [&](uint64_t k) {
            emit_slot<double, true, false>(&batch, lane, geos, offs, C.n_geoms, k, M, nullptr, key, 0.0);
          },
          [&](unsigned slot, uint64_t) {
            batch.load(slot, p, M, nullptr);
            if (p.g != acct.g) {
              acct.flush(A);
              acct.reset(p.g);
            }
            G = &geos[p.g];
            if (CELLS) {
              T.cP = A.cellP + (copy * C.n_geoms + p.g) * C.n_cells * 4;
              T.h = G->L[C.cell_axis] / (double)C.n_cells;
              T.inv_h = (float)C.n_cells / G->Lf[C.cell_axis];
            }
            T.qb = C.per_bin ? A.qbin + (copy * C.n_geoms + p.g) * M.n : nullptr;
            T.det = C.n_regs > 0 ? A.det_raw : nullptr;
            if (GRAD) gr.init(p.bin);
            alive = true;
          });
    }
    if (!__any_sync(kAll, alive)) {
      if (pool_dry) break;
      continue;
    }
    if (!alive) continue;
    int out = step_steady<double, GradT, TallyPlain>(p, *G, M, M.rec_relax, nullptr, C, key.x, key.y, T, gr);
    if (out == STEP_ALIVE && (p.e & 1023u) == 0u && globaltimer_ns() > deadline) {
      atomicOr(A.flags, 1);
      out = STEP_TRUNCATED;
    }
    if (out == STEP_ALIVE) continue;
    if constexpr (GRAD) {
      if (gr.mv.phase) {   // the phantom trace: nothing is tallied but its X
        const double D = gr.mv.score(X_nom, p.X);
        double* gs = grad_copy(A);
        atomicAdd(gs + 1, D);
        atomicAdd(gs + 2, D * D);
        alive = false;
        continue;
      }
    }
    T.period_end(p);
    acct.end(out, p.e + 1u, p.s > 0.0 ? 1 : -1, p.X, p.X);
    if (A.events_pp || A.X_pp) {
      const uint64_t idx = offs[p.g] + (p.pid - (uint32_t)G->pid0);
      if (A.events_pp) A.events_pp[idx] = p.e + 1u;
      if (A.X_pp) A.X_pp[idx] = p.X;
    }
    nscat_end(C, p.g, p.n_relax, p.X);
    alive = false;
    if constexpr (GRAD) {
      grad_finish(gr, p.X, p.g, C, A, M);
      if (C.mvd && gr.mv.sel > 0u) {
        // measure-valued d/dp_pore: the particle again from its emission, the
        // chosen pore hit's branch flipped
        X_nom = p.X;
        gr.mv.start_phantom();
        T.cP = T.qb = T.det = nullptr;
        emit<double>(p, *G, M, M.rec_emit, M.rec_init, nullptr, key.x, key.y, false, 0.0);
        alive = true;
      }
    }
  }
  if (C.n_geoms == 1) s_acct.add(acct);
  else acct.flush(A);
  __syncthreads();
  if (threadIdx.x == 0 && C.n_geoms == 1) s_acct.flush(A);
}
#endif  // MCBTE_F64

#if MCBTE_F32
// ------------------------------------------------------------------ FP32 persistent
// Gradient pass: the open period closes at the particle's end (X = X_f; a
// fused pass adds its listed periods' a X_f too), then the resampling and
// specularity terms and the directional values.
__device__ __forceinline__ void grad_finish_replay(GradReplay& gr, double X, int g, const RunCfg& C, const Acc& A) {
  gr.finish(X);
  const double Rv = gr.resample_term(X);
  double* gs = grad_copy(A);
  atomicAdd(gs + 0, Rv);
  if (!C.mvd) {   // the measure-valued score is added after the phantom trace
    const double gp = gr.spec_term(X);
    atomicAdd(gs + 1, gp);
    atomicAdd(gs + 2, gp * gp);
  }
  for (int kd = 0; kd < C.n_dirs; ++kd) {
    const double val = gr.dv[kd] + Rv * C.dpi[kd];
    atomicAdd(gs + 4 + 2 * kd, val);
    atomicAdd(gs + 5 + 2 * kd, val * val);
  }
}

// A particle the main FP32 kernel hands to the tail kernel: the state the
// FP32 steady step carries (v, 1/v and Lambda are the bin's, reloaded), its
// index in the run and, in the gradient pass, the gradient bookkeeping.  Only
// these fields are stored, so parking keeps nothing else alive in the loop.
struct ParkRec {
  int4 snap[4];   // gradient pass: the pore-hit snapshot (snap_ok)
  float x[3], u[3], d_rel, d2, s;
  int bin, n_relax, g;
  uint32_t e, pid;
  long long Xq, Xqper;
  // gradient pass
  double Xf, sum_x_res;
  float a, d, pa, pd;
  int bin_cur, n_res;
  uint32_t mK, mKn, msel;
  int mflags;   // bit 0 sel_spec, bit 1 phase
  double dv[kMaxDirs];
  int np;       // fused gradient pass: the listed periods
  int lb[kFusedPeriods];
  float la[kFusedPeriods];
  int snap_ok;
};

template <bool GRAD, class GradT>
__device__ __forceinline__ void park_store(ParkRec* r, const Particle<float>& p, const GradT& gr,
                                           int n_dirs) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    r->x[a] = p.x[a];
    r->u[a] = p.u[a];
  }
  r->d_rel = p.d_rel;
  r->d2 = p.d2;
  r->s = p.s;
  r->bin = p.bin;
  r->n_relax = p.n_relax;
  r->g = p.g;
  r->e = p.e;
  r->pid = p.pid;
  r->Xq = p.Xq;
  r->Xqper = p.Xqper;
  if constexpr (GRAD) {
    r->Xf = gr.Xf;
    r->sum_x_res = gr.sum_x_res;
    r->a = gr.a;
    r->d = gr.d;
    r->pa = gr.pa;
    r->pd = gr.pd;
    r->bin_cur = gr.bin_cur;
    r->n_res = gr.n_res;
    r->mK = gr.mv.K;
    r->mKn = gr.mv.Kn;
    r->msel = gr.mv.sel;
    r->mflags = (gr.mv.sel_spec ? 1 : 0) | (gr.mv.phase ? 2 : 0);
    for (int k = 0; k < n_dirs; ++k) r->dv[k] = gr.dv[k];
    r->np = gr.np;
    for (int k = 0; k < gr.np; ++k) {
      r->lb[k] = gr.lb[k];
      r->la[k] = gr.la[k];
    }
    r->snap_ok = gr.snap_ok ? 1 : 0;
    if (gr.snap_ok) {
#pragma unroll
      for (int k = 0; k < 4; ++k) r->snap[k] = gr.snap[k];
    }
  }
}

template <bool GRAD, class GradT>
__device__ __forceinline__ void park_load(const ParkRec* r, Particle<float>& p, GradT& gr, int n_dirs,
                                          const MatView& M, const float4* binf) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    p.x[a] = r->x[a];
    p.u[a] = r->u[a];
  }
  p.d_rel = r->d_rel;
  p.d2 = r->d2;
  p.s = r->s;
  p.bin = r->bin;
  p.n_relax = r->n_relax;
  p.g = r->g;
  p.e = r->e;
  p.pid = r->pid;
  p.Xq = r->Xq;
  p.Xqper = r->Xqper;
  load_bin(p, M, binf);
  if constexpr (GRAD) {
    gr.Xf = r->Xf;
    gr.sum_x_res = r->sum_x_res;
    gr.a = r->a;
    gr.d = r->d;
    gr.pa = r->pa;
    gr.pd = r->pd;
    gr.bin_cur = r->bin_cur;
    gr.n_res = r->n_res;
    gr.mv.K = r->mK;
    gr.mv.Kn = r->mKn;
    gr.mv.sel = r->msel;
    gr.mv.sel_spec = (r->mflags & 1) != 0;
    gr.mv.phase = (r->mflags & 2) != 0;
    for (int k = 0; k < n_dirs; ++k) gr.dv[k] = r->dv[k];
    gr.np = r->np;
    for (int k = 0; k < gr.np; ++k) {
      gr.lb[k] = r->lb[k];
      gr.la[k] = r->la[k];
    }
    // without a snapshot here the phantom trace starts from the emission
    gr.snap_ok = r->snap_ok != 0 && gr.snap != nullptr;
    if (gr.snap_ok) {
#pragma unroll
      for (int k = 0; k < 4; ++k) gr.snap[k] = r->snap[k];
    }
  }
}

// The tail kernel's events of one live particle from its precomputed draws
// where trace_lean does not go (extended physics with detector regions, the
// N_scat_max curve, or walls in a batch of geometries): slot0 holds the draws
// of event p.e + 1, and the slots end with event e_last.  Returns at the
// particle's end, or ALIVE once the slots are used up.
template <class Grad, class Tally>
__device__ __forceinline__ int trace_slots(Particle<float>& p, const GeoRun& g, const MatView& M, const uint4* relax_tab,
                                           const float4* binf, const RunCfg& C, uint32_t k0, uint32_t k1,
                                           const Tally& T, Grad& gr, const DrawLean* slot0, uint32_t e_last) {
  const uint32_t e0 = p.e;
  for (;;) {
    const int out = step_steady<float, Grad, Tally, true, DrawSlot>(p, g, M, relax_tab, binf, C, k0, k1, T, gr,
                                                                    DrawSlot{slot0 + (p.e - e0)});
    if (out != STEP_ALIVE) return out;
    if (p.e >= e_last) return STEP_ALIVE;
  }
}

// The tail loop of a particle whose flights run through unfolded periodic
// axes (forward run without cell tallies or extended physics; a box with no
// pore and no walls): trace_slots with step_steady's unfolded flight.  The
// crossings advance the event number, so the event that ends a flight may
// lie past the slots and then takes its draws inline (the same bits).
template <class Tally>
__device__ __forceinline__ int trace_unfolded(Particle<float>& p, const GeoRun& g, const MatView& M,
                                              const uint4* relax_tab, const float4* binf, const RunCfg& C, uint32_t k0,
                                              uint32_t k1, const Tally& T, const DrawLean* slot0, uint32_t e_last,
                                              unsigned um) {
  const uint32_t e0 = p.e;
  const uint32_t nslots = e_last - e0;
  GeoLean gl;
  gl.load(g);
  GradOff off;
  for (;;) {
    if (p.e + 1u >= C.max_events) return STEP_TRUNCATED;
    float db;
    int face;
    hit_box_pore_f32(gl, p.x, p.u, &db, &face, um);
    const bool relax = p.d_rel < db;
    const float seg = relax ? p.d_rel : db;
    T.segment(p, seg);
#pragma unroll
    for (int a = 0; a < 3; ++a) p.x[a] = p.x[a] + seg * p.u[a];
    const uint32_t n = fold_periodic(p.x, gl.Lf, um);
    if (n >= C.max_events - 1u - p.e) {
      p.e = C.max_events - 1u;
      return STEP_TRUNCATED;
    }
    p.e += n;
    const uint32_t si = p.e - e0;
    const Draw32* slot = si < nslots ? slot0 + si : nullptr;
    if (!relax && face < 6) {
      // apply_event's FP32 face branch (every periodic axis is unfolded, so
      // the face is isothermal: absorbed, or adiabatic: specular or
      // Lambertian by the event's draws, then a select)
      ++p.e;
      p.d_rel = p.d_rel - seg;
      const int a = face_axis(face);
      const int mx = face_is_max(face);
      put3<float>(p.x, a, mx ? gl.L(a) : 0.0f);
      if (gl.type(face) == MCBTE_FACE_ISOTHERMAL) return STEP_ABSORBED;
      const Draw32 d = DrawSlotOr{slot}.sub0(make_uint4(p.pid, (uint32_t)p.g, p.e, 0u), k0, k1, relax_tab, M.n);
      const bool spec_f = (uint64_t)d.wx < g.pthr[face];
      float ud[3];
      put3_cyclic<float>(ud, a, mx ? -d.lam[0] : d.lam[0], d.lam[1], d.lam[2]);
      const float flip = -sel3(p.u, a);
#pragma unroll
      for (int b = 0; b < 3; ++b) p.u[b] = spec_f ? (b == a ? flip : p.u[b]) : ud[b];
    } else {
      const int out = apply_event<float, GradOff, Tally, false, DrawSlotOr>(p, g, M, relax_tab, binf, C, k0, k1,
                                                                            relax, false, face, seg, T, off, 0.0,
                                                                            DrawSlotOr{slot});
      if (out != STEP_ALIVE) return out;
    }
    if (p.e >= e_last) return STEP_ALIVE;
  }
}

// Every lane owns one particle at a time.  When its particle terminates the
// lane refills from its warp's batch (Refill: 32 particles emitted at once by
// all lanes into shared memory, from the warp's run of particle indices, which
// is refilled from the global work counter a chunk at a time).  Lanes therefore
// never idle while work remains, whatever the event-count spread between
// particles, and the emission runs with all lanes.  Emitting for the waiting
// lanes alone took 150 warp instructions a particle; what made room for the
// batch at 80 registers a thread is that nothing a particle needs once (the
// lane's book-keeping, the warp's run) stays in registers.  1e7-particle
// silicon-like slab: 17.98 -> 15.32 ms.  Blocks of 1024 threads have 64
// registers, which the batch made the event loop spill, and the batches' room
// is the L1's: their lanes emit for themselves (kUnbatchedThreads).
// TPB is the block size the kernel is compiled for (register budget).
// GRAD: the gradient pass.  Fused (C.fused): the forward run's tallies,
// counters and per-particle outputs and the gradient in one pass, each
// particle listing its periods until its final tally is known.  Otherwise
// the replay of the forward pass's particles with their final tallies read
// from A.X_pp: it writes the gradient accumulators only, and flags (bit 2)
// any particle whose replayed tally differs.  With the measure-valued
// d/dp_pore the lane then traces the same particle once more (phantom
// phase, the chosen pore hit flipped, resumed from the lane's snapshot of
// that hit where it has one) before it refills.
// UNF (no cell tallies, no extended physics, no gradient): flights run
// through the periodic faces of a box without pore or walls (step_steady).
// CELLS: 0 no cell tallies, 1 T and three flux components, 2 T and the
// tally-axis flux only.
//
// MODE 0: the main kernel of a run without the tail kernel.  The run's tail
// (MODE 1 and 2): once the work counter has run out, a warp of the main
// kernel (MODE 1) with at most C.tail_max particles in flight parks them
// (ParkRec, A.park) and retires, so no warp idles most of its lanes for the
// rest of the run.  The tail kernel (MODE 2, launched next on the same
// stream) takes the parked particles instead of emitting new ones; once none
// is left, a warp with at most C.tail_max particles in flight computes the
// draws of their next events on all 32 lanes at once (two DrawLean per lane,
// the warp's 64 slots shared out over its live particles, 64 / 2^ceil(log2
// live) events each) and every live lane traces that many events reading its
// slots (tail.cuh), so its dependent chain per event holds the geometry and
// the tallies only.  The draws are the inline path's, the parked state is
// resumed as it was: trajectories and tallies are bit for bit those of a
// single kernel.
template <int CELLS, bool GRAD, int TPB, bool EXT, int MODE>
__global__ void __launch_bounds__(TPB, 1) k_steady_f32(const GeoRun* __restrict__ geos,
                                                       const uint64_t* __restrict__ offs, MatView M, RunCfg C,
                                                       Acc A, SmemPlan S) {
  constexpr bool TK = MODE == 2;
  // flights through the unfolded periodic axes (step_steady)
  constexpr bool UNF = CELLS == 0 && !GRAD && !EXT;
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned char* sp = smem;
  const int n = M.n;
  const int nc = C.n_cells;
  const uint4* relax = M.rec_relax;
  const float4* binf = M.binf;
  long long* s_qbin = nullptr;
  long long* s_cP = nullptr;
  long long* s_cD = nullptr;
  // the warps' emitted batches (main kernel) or the tail kernel's draw slots
  // come first (16-byte aligned)
  constexpr bool kBatched = !TK && TPB < kUnbatchedThreads;
  using BatchT = EmitBatch<float, EXT, false>;
  Refill& refill = reinterpret_cast<Refill*>(sp)[threadIdx.x >> 5];
  const unsigned slot_at = (threadIdx.x >> 5) * (unsigned)S.batch_slots;   // the warp's first, over all records
  BatchT& batch = reinterpret_cast<BatchT*>(sp + (TPB / 32) * sizeof(Refill))[slot_at / kBatchSlots];
  const unsigned slot0 = slot_at % kBatchSlots;
  if constexpr (kBatched)
    sp += (TPB / 32) * sizeof(Refill) + ((TPB / 32) * (unsigned)S.batch_slots / kBatchSlots) * sizeof(BatchT);
  DrawLean* slots = nullptr;
  if (TK) {
    slots = reinterpret_cast<DrawLean*>(sp) + (size_t)(threadIdx.x >> 5) * S.tail_slots;
    sp += (size_t)(TPB / 32) * S.tail_slots * sizeof(DrawLean);
  }
  // then the pore-hit snapshots (16-byte aligned), four int4 per thread
  int4* snaps = nullptr;
  if (S.snap_in_smem) {
    snaps = reinterpret_cast<int4*>(sp) + (size_t)threadIdx.x * 4;
    sp += (size_t)TPB * 4 * sizeof(int4);
  }
  if (S.relax_in_smem) {
    uint4* t = reinterpret_cast<uint4*>(sp);
    for (int i = threadIdx.x; i < n; i += blockDim.x) t[i] = M.rec_relax[i];
    relax = t;
    sp += (size_t)n * sizeof(uint4);
  }
  if (S.binf_in_smem) {
    float4* t = reinterpret_cast<float4*>(sp);
    for (int i = threadIdx.x; i < n; i += blockDim.x) t[i] = M.binf[i];
    binf = t;
    sp += (size_t)n * sizeof(float4);
  }
  if (S.qbin_in_smem) {
    s_qbin = reinterpret_cast<long long*>(sp);
    for (int i = threadIdx.x; i < n; i += blockDim.x) s_qbin[i] = 0;
    sp += (size_t)n * sizeof(long long);
  }
  long long* s_grad = nullptr;
  if (S.grad_in_smem) {
    s_grad = reinterpret_cast<long long*>(sp);
    for (int i = threadIdx.x; i < n; i += blockDim.x) s_grad[i] = 0;
    sp += (size_t)n * sizeof(long long);
  }
  if (S.cells_in_smem) {
    s_cP = reinterpret_cast<long long*>(sp);
    s_cD = s_cP + (size_t)nc * 4;
    for (int i = threadIdx.x; i < nc * 4 + (nc + 1) * 4; i += blockDim.x) s_cP[i] = 0;
  }
  __shared__ BlockAcct<long long> s_acct;
  if (threadIdx.x == 0) s_acct.reset();
  // the tail's walls (one geometry)
  __shared__ WallLean s_walls[TK && EXT ? kMaxInner : 1];
  if (TK && EXT && C.n_geoms == 1)
    for (int i = threadIdx.x; i < kMaxInner; i += blockDim.x) s_walls[i].set(geos[0], i);
  __syncthreads();

  const unsigned lane = threadIdx.x & 31u;
  const uint64_t deadline = *C.t0 + C.budget_ns;
  Particle<float> p;
  using GradT = typename GradPick<GRAD, GradReplay>::type;
  GradT gr;
  double gr_dv[GRAD ? kMaxDirs : 1];
  int gr_lb[GRAD ? kFusedPeriods : 1];
  float gr_la[GRAD ? kFusedPeriods : 1];
  if constexpr (GRAD) {
    gr.dv = gr_dv;
    gr.lb = gr_lb;
    gr.la = gr_la;
    gr.snap = snaps;
    gr.G = S.grad_in_smem ? s_grad : A.Gq;
    gr.fused = C.fused != 0;
    gr.n_dirs = C.n_dirs;
    gr.n_bins = n;
    gr.dirs = C.dirs;
    gr.mvd = C.mvd != 0;
    gr.sc_spec = (float)(1.0 / geos[0].p_pore);
    gr.sc_diff = (float)(-1.0 / (1.0 - geos[0].p_pore));
  }
  // The lane's book-keeping is touched once per particle: kept in local memory
  // (an address the compiler cannot see through), its 13 registers go to the
  // event loop.
  ThreadAcct<long long> acct;
  acct.reset(-1);
  auto acct_mem = [&]() -> ThreadAcct<long long>* {
    ThreadAcct<long long>* q = &acct;
    // (no instruction: hides where q points)
    asm volatile("" : "+l"(q) : : "memory");
    return q;
  };
  TallyFxT<CELLS == 2 ? 2 : 4> T;
  T.nc = nc;
  T.ca = C.cell_axis;
  T.ta = C.tally_axis;
  T.cP = T.cD = T.qb = nullptr;
  T.h = T.inv_h = 1.0f;
  T.det = (C.n_regs > 0 && !GRAD) ? A.det_q : nullptr;
  // the per-bin flux of the particle's geometry (a gradient pass tallies
  // only when fused, and never in a phantom trace)
  auto qbin_of = [&](int g) -> long long* {
    if (!C.per_bin || (GRAD && !C.fused)) return nullptr;
    return S.qbin_in_smem ? s_qbin : A.qbinq + (size_t)g * n;
  };
  bool alive = false;
  bool drained = false;   // no work left for this lane: it idles in the loop until its warp is drained
  const GeoRun* G = geos;
  const uint2 key = run_key(C);
  const int refill_min = (C.refill_min > 1 && !TK) ? C.refill_min : 1;
  // the tail: parking (main kernel) or the draws ahead (tail kernel)
  const int tail_max = (TK ? n <= kOneBlockBins : (MODE == 1 && A.park_cap > 0)) ? C.tail_max : 0;
  const uint64_t n_parked = TK ? min(*(volatile unsigned long long*)A.park_n, (unsigned long long)A.park_cap) : 0;
  bool pool_dry = false;   // the same in every lane: nothing left to hand out
  WarpRun run;   // without a batch: the warp's particle indices not yet handed out
  if constexpr (kBatched) refill.start(lane, C.take_chunk, C.total, deadline, A.flags);
  else if constexpr (!TK) run.start(C.take_chunk, C.total, deadline, A.flags);
  // a particle's index in the run
  auto index_of = [&](const Particle<float>& q) { return offs[q.g] + (q.pid - (uint32_t)geos[q.g].pid0); };
  // the tallies of the lane's geometry
  auto bind = [&](int g) {
    ThreadAcct<long long>* am = acct_mem();
    if (g != am->g) {
      am->flush(A);
      am->reset(g);
    }
    G = &geos[g];
    if (CELLS) {
      T.cP = S.cells_in_smem ? s_cP : A.cellPq + (size_t)g * nc * 4;
      T.cD = S.cells_in_smem ? s_cD : A.cellDq + (size_t)g * (nc + 1) * 4;
      T.h = G->Lf[C.cell_axis] / (float)nc;
      T.inv_h = (float)nc / G->Lf[C.cell_axis];
    }
    T.qb = qbin_of(g);
  };
  // All 32 lanes stay in the loop until every lane of the warp is drained, so
  // the warp-wide votes below reconverge the warp at every event step.
  constexpr unsigned kAll = 0xffffffffu;
  for (;;) {
    // two votes per step: the drained lanes and the busy ones
    const unsigned dry = __ballot_sync(kAll, drained);
    if (dry == kAll) break;
    const unsigned live = __ballot_sync(kAll, alive);
    const int nlive = __popc(live);
    int out = STEP_ALIVE;
    if (MODE != 0 && pool_dry && nlive > 0 && nlive <= tail_max) {
      if constexpr (MODE == 1) {
        // park the warp's last particles for the tail kernel
        const int leader = __ffs(live) - 1;
        unsigned long long base = 0;
        if ((int)lane == leader) base = atomicAdd(A.park_n, (unsigned long long)nlive);
        base = __shfl_sync(kAll, base, leader);
        if (alive) {
          const unsigned long long slot = base + (unsigned long long)__popc(live & ((1u << lane) - 1u));
          if (slot < A.park_cap) {
            park_store<GRAD>(reinterpret_cast<ParkRec*>(A.park + slot * A.park_stride), p, gr, C.n_dirs);
            alive = false;
            drained = true;
          }
        }
        continue;   // lanes the buffer could not take trace on with the next votes (park_cap reached)
      } else {
        // log2 of the slots per particle: nlive << sh <= S.tail_slots
        const int sh = (31 - __clz(S.tail_slots)) - (32 - __clz(nlive - 1));
        const unsigned um = (UNF && alive) ? unfold_mask<GradT>(*G, C) : 0u;
        // draws ahead, or (most of the live particles in thick films) inline
        bool ahead = true;
        float per_flight = 0.0f;
        if constexpr (UNF) {
          if (alive) per_flight = film_events(*G, um);
          const bool inl = per_flight * kInlineFlights > (float)(1u << sh);
          ahead = 2 * __popc(__ballot_sync(kAll, alive && inl)) <= nlive || __any_sync(kAll, alive && per_flight == 0.0f);
        }
#pragma unroll
        for (int h = 0; h < kTailSlots / 32; ++h) {
          if (!ahead || 32 * h >= S.tail_slots) break;
          const unsigned i = lane + 32u * h;
          const int r = (int)(i >> sh);   // the live particle slot i belongs to
          // its lane: a lone particle's is the only one, else the r-th live lane
          unsigned mm = live;
          if (nlive > 1)
            for (int k = 0; k < r && mm; ++k) mm &= mm - 1u;
          const int owner = mm ? __ffs(mm) - 1 : 0;
          const uint32_t e_o = __shfl_sync(kAll, p.e, owner);
          const uint32_t pid_o = __shfl_sync(kAll, p.pid, owner);
          const int g_o = __shfl_sync(kAll, p.g, owner);
          float s_o = 0.0f;
          if constexpr (UNF) s_o = __shfl_sync(kAll, p.s, owner);
          if (r < nlive) {
            DrawLean d;
            uint4 ctr = make_uint4(pid_o, (uint32_t)g_o, e_o + 1u + (i & ((1u << sh) - 1u)), 0u);
            draw_words(d, philox(ctr, key.x, key.y), relax, n);
            d.E2 = 0.0f;
            d.mv_lo = d.mv_hi = 0u;
            if (EXT && M.imp) {
              ctr.w = 256u;
              d.E2 = draw_e2(philox(ctr, key.x, key.y));
            }
            if (GRAD && C.mvd) {
              ctr.w = 257u;
              const uint4 w7 = philox(ctr, key.x, key.y);
              d.mv_lo = w7.x;
              d.mv_hi = w7.y;
            }
            draw_lean(d, geos[g_o], binf, EXT);
            if constexpr (UNF) {
              const unsigned um_o = unfold_mask<GradT>(geos[g_o], C);
              const int W = um_o == 3u ? 2 : (um_o == 5u ? 1 : (um_o == 6u ? 0 : -1));
              if (W >= 0) d.to_film(geo_L<float>(geos[g_o], W), W, s_o, T.ta);
            }
            slots[i] = d;
          }
        }
        __syncwarp();
        if (alive) {
          const DrawLean* s0 = slots + (__popc(live & ((1u << lane) - 1u)) << sh);
          const uint32_t e_f = p.e, nslots = ahead ? 1u << sh : 0u;
          const uint32_t e_l =
              round_end(p.e, ahead ? nslots : (uint32_t)fminf(kInlineRound * per_flight, 65536.0f), C.max_events);
          const bool film = um == 3u || um == 5u || um == 6u;
          if (UNF && um && !film) {
            out = trace_unfolded(p, *G, M, relax, binf, C, key.x, key.y, T, s0, e_l, um);
          } else if (EXT && (C.n_regs > 0 || C.nscat_acc || (C.n_geoms > 1 && G->n_inner > 0))) {
            out = trace_slots<GradT, decltype(T)>(p, *G, M, relax, binf, C, key.x, key.y, T, gr, s0, e_l);
          } else {
            const LoneArgs la{C.max_events, C.n_scat_max, n, M.imp, M.spec_thr, relax, binf, key.x, key.y};
            out = trace_alone<GradT, decltype(T), EXT, (CELLS > 0)>(p, *G, s_walls, la, T, gr, s0, nslots, e_l, um);
          }
          // (the time budget every 256 events)
          if (out == STEP_ALIVE && ((e_f ^ p.e) >> 8) != 0u && globaltimer_ns() > deadline) {
            atomicOr(A.flags, 1);
            out = STEP_TRUNCATED;
          }
        }
        __syncwarp();   // the slots are rewritten in the next round
      }
    } else {
      const unsigned need = ~(dry | live);
      // refill once enough lanes are idle (or no lane is busy)
      if (need && !pool_dry && (__popc(need) >= refill_min || live == 0u)) {
        if constexpr (TK) {
          const unsigned cnt = __popc(need);
          const unsigned rank = __popc(need & ((1u << lane) - 1u));
          const int leader = __ffs(need) - 1;
          unsigned long long base = 0;
          if ((int)lane == leader) base = atomicAdd(A.park_rd, (unsigned long long)cnt);
          base = __shfl_sync(kAll, base, leader);
          if (base + cnt >= n_parked) pool_dry = true;
          const uint64_t k = base + rank;
          if (!alive && !drained) {
            if (k >= n_parked || (*(volatile int*)A.flags & 1)) {
              drained = true;
              continue;
            }
            // a parked particle, exactly as the main kernel left it
            park_load<GRAD>(reinterpret_cast<const ParkRec*>(A.park + k * A.park_stride), p, gr, C.n_dirs, M,
                            binf);
            bind(p.g);
            if constexpr (GRAD) {
              if (gr.mv.phase) T.qb = nullptr;   // a phantom trace tallies only its own X
            }
            alive = true;
          }
        } else if constexpr (!kBatched) {
          const uint64_t k = run.take(need, lane, A.work, C.total, deadline, A.flags);
          if (run.empty()) pool_dry = true;
          if (!alive && !drained) {
            if (k >= C.total || (*(volatile int*)A.flags & 1)) {
              drained = true;
              continue;
            }
            const int g = find_geom(offs, C.n_geoms, k);
            bind(g);
            p.pid = (uint32_t)(k - offs[g] + G->pid0);
            p.g = g;
            emit<float, EXT>(p, *G, M, M.rec_emit, M.rec_init, binf, key.x, key.y, false, 0.0f);
            if constexpr (GRAD) {
              gr.init(p.bin);
              if (!C.fused) gr.Xf = A.X_pp[k];
            }
            alive = true;
          }
        } else {
          pool_dry = refill.hand_out(
              S.batch_slots, need, lane, A.work, C.total, deadline, A.flags,
              [&](uint64_t k) {
                emit_slot<float, EXT, false>(&batch, slot0 + lane, geos, offs, C.n_geoms, k, M, binf, key, 0.0f);
              },
              [&](unsigned slot, uint64_t k) {
                batch.load(slot0 + slot, p, M, binf);
                bind(p.g);
                if constexpr (GRAD) {
                  gr.init(p.bin);
                  if (!C.fused) gr.Xf = A.X_pp[k];
                }
                alive = true;
              });
        }
      }
      if (!alive) {
        drained = drained || pool_dry;   // nothing left to hand out
        continue;
      }
      out = step_steady<float, GradT, decltype(T), EXT, DrawInline, UNF>(p, *G, M, relax, binf, C, key.x, key.y, T,
                                                                          gr);
      if (out == STEP_ALIVE && (p.e & 255u) == 0u && globaltimer_ns() > deadline) {
        atomicOr(A.flags, 1);
        out = STEP_TRUNCATED;
      }
    }
    if (!alive || out == STEP_ALIVE) continue;
    // the forward run's part of a finished (nominal) trace: the last period's
    // per-bin flux, the run's counters and sums, the per-particle outputs
    auto account = [&](double X) {
      T.period_end(p);
      const unsigned nev = p.e + 1u;
      // one read and write of the lane's fields, which live in memory (below)
      ThreadAcct<long long> t = *acct_mem();
      t.end(out, nev, p.s > 0.0f ? 1 : -1, p.Xq, X);
      *acct_mem() = t;
      if (A.events_pp) A.events_pp[index_of(p)] = nev;
      if (A.X_pp) A.X_pp[index_of(p)] = X;
      if constexpr (EXT) nscat_end(C, p.g, p.n_relax, X);
    };
    if (GRAD) {
      const double X = T.X(p);
      if constexpr (GRAD) {
        if (!gr.mv.phase) {
          if (C.fused) account(X);
          else if (X != gr.Xf) atomicOr(A.flags, 4);
          grad_finish_replay(gr, X, p.g, C, A);
          if (C.mvd && gr.mv.sel > 0u) {
            // measure-valued d/dp_pore: the same particle again from its
            // emission, the chosen pore hit's branch flipped (Xf keeps the
            // nominal tally; the phantom tallies only its own X)
            gr.Xf = X;
            gr.mv.start_phantom();
            T.qb = nullptr;
            if (gr.snap_ok) {
              // resume at the chosen hit (the state the trace from the
              // emission would reach) and apply it with its branch flipped
              gr.restore(p);
              load_bin(p, M, binf);
              gr.mv.K = gr.mv.sel - 1u;
              apply_event<float, GradT, decltype(T), EXT>(p, *G, M, relax, binf, C, key.x, key.y, false, false, 6,
                                                          0.0f, T, gr, T.X(p));
            } else {
              emit<float, EXT>(p, *G, M, M.rec_emit, M.rec_init, binf, key.x, key.y, false, 0.0f);
            }
            continue;
          }
        } else {
          const double D = gr.mv.score(gr.Xf, X);
          double* gs = grad_copy(A);
          atomicAdd(gs + 1, D);
          atomicAdd(gs + 2, D * D);
        }
      }
    } else {
      account(T.X(p));
    }
    alive = false;
    drained = pool_dry;
  }
  const bool one_geom = C.n_geoms == 1;
  if (!GRAD || C.fused) {
    if (one_geom) s_acct.add(*acct_mem());
    else acct_mem()->flush(A);
  }
  __syncthreads();
  if (threadIdx.x == 0 && one_geom) s_acct.flush(A);
  if (S.qbin_in_smem) {
    for (int i = threadIdx.x; i < n; i += blockDim.x)
      if (s_qbin[i] != 0) atomicAdd(reinterpret_cast<unsigned long long*>(&A.qbinq[i]), (unsigned long long)s_qbin[i]);
  }
  if (S.grad_in_smem) {
    for (int i = threadIdx.x; i < n; i += blockDim.x)
      if (s_grad[i] != 0) atomicAdd(reinterpret_cast<unsigned long long*>(&A.Gq[i]), (unsigned long long)s_grad[i]);
  }
  if (S.cells_in_smem) {
    for (int i = threadIdx.x; i < nc * 4; i += blockDim.x)
      if (s_cP[i] != 0) atomicAdd(reinterpret_cast<unsigned long long*>(&A.cellPq[i]), (unsigned long long)s_cP[i]);
    for (int i = threadIdx.x; i < (nc + 1) * 4; i += blockDim.x)
      if (s_cD[i] != 0) atomicAdd(reinterpret_cast<unsigned long long*>(&A.cellDq[i]), (unsigned long long)s_cD[i]);
  }
}
#endif  // MCBTE_F32

#if MCBTE_F64
// ------------------------------------------------------------------ finalise
// One block per geometry: scale the raw sums into the paper's estimators
// (Eqs. temp_steady, flux_x_steady), kappa = -q / (dT/dx) and its standard
// error from the per-particle X_p (iid), and the LR gradient.  FP64 and
// fixed-point accumulators are both read (only one kind is non-zero).
__global__ void k_finalize_steady(const GeoRun* geos, MatView M, RunCfg C, Acc A, SteadyOutDev O, int grad,
                                  const int* flags) {
  const int g = blockIdx.x;
  const GeoRun& G = geos[g];
  const int nc = C.n_cells;
  const int n = M.n;
  const double N = (double)G.n_norm;
  const double E_eff = G.E_tot / N;
  const double C_tot = M.sums[0];
  const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  if (nc > 0 && warp < 4) {
    // cells: warp b takes component b (T, q_x, q_y, q_z) of all cells, the
    // difference array folded by a warp scan of the integer sums, 32 cells at
    // a time (one thread over all cells and components took 68 us for 50
    // cells, all of it load latency; the kernel now takes 6 us)
    const int b = (int)warp;
    const double Vc = G.V_box / (double)nc;
    const double k = b == 0 ? E_eff / (C_tot * Vc) : E_eff / Vc;
    const size_t stride = (size_t)C.n_geoms * nc * 4;   // between copies (FP64 path)
    long long carry = 0;
    for (int c0 = 0; c0 < nc; c0 += 32) {
      const int c = c0 + (int)lane;
      const bool in = c < nc;
      double v = 0.0;
      if (C.f64_rep) {
        if (in) {
          const double* P = A.cellP + ((size_t)g * nc + c) * 4 + b;
#pragma unroll 8
          for (int r = 0; r < C.f64_rep; ++r) v += P[r * stride];
        }
      } else {
        const size_t at = ((size_t)g * nc + c) * 4 + b;
        long long run = in ? A.cellDq[at + (size_t)g * 4] : 0;   // [G][nc + 1][4]
        const long long pq = in ? A.cellPq[at] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const long long y = __shfl_up_sync(0xffffffffu, run, o);
          if ((int)lane >= o) run += y;
        }
        run += carry;
        carry = __shfl_sync(0xffffffffu, run, 31);
        v = (double)(pq + run) * kFxInv;
      }
      if (!in) continue;
      if (b == 0 && O.T) O.T[(size_t)g * nc + c] = (k * v) * 1e-12;
      if (b > 0 && O.q) O.q[((size_t)g * nc + c) * 3 + (b - 1)] = (k * v) * 1e-9;
    }
  }
  if (O.det && C.n_regs > 0) {
    // detector regions: volume-averaged T and q of each detector (and bin)
    const double C_tot_d = M.sums[0];
    const size_t nb = C.det_nb > 1 ? (size_t)C.det_nb : 1;
    for (size_t s = threadIdx.x; s < (size_t)C.n_det * nb; s += blockDim.x) {
      const uint32_t d = (uint32_t)(s / nb);
      double vd = C.regs[0].v_det;
      for (int k = 0; k < C.n_regs; ++k)
        if (d >= C.regs[k].off) vd = C.regs[k].v_det;
      const double kT = E_eff / (C_tot_d * vd);
      const double kq = E_eff / vd;
      double raw[4];
      for (int b = 0; b < 4; ++b) raw[b] = A.det_raw[s * 4 + b] + (double)A.det_q[s * 4 + b] * kFxInv;
      O.det[s * 4 + 0] = (kT * raw[0]) * 1e-12;
      for (int b = 1; b < 4; ++b) O.det[s * 4 + b] = (kq * raw[b]) * 1e-9;
    }
  }
  if (O.kn && C.nscat_acc) {
    // fold the copies of the curve sums into the first
    const size_t per = (size_t)(C.n_scat_max + 1) * 4;
    const size_t stride = (size_t)C.n_geoms * per;
    double* a0 = C.nscat_acc + (size_t)g * per;
    for (size_t i = threadIdx.x; i < per; i += blockDim.x) {
      double v = a0[i];
      for (int r = 1; r < C.nscat_rep; ++r) v += a0[(size_t)r * stride + i];
      a0[i] = v;
    }
    __syncthreads();
  }
  if (O.kn && C.nscat_acc && threadIdx.x == 0) {
    // kappa and its standard error for N_scat_max = k: the tally at the k-th
    // relaxation, or the final one of trajectories that ended before it
    const int K = C.n_scat_max;
    const double nt = (double)A.cnt[g * 4 + 3];
    const double* a = C.nscat_acc + (size_t)g * (size_t)(K + 1) * 4;
    double e1 = 0.0, e2 = 0.0;
    for (int k = 1; k <= K; ++k) {
      e1 += a[(size_t)k * 4 + 2];
      e2 += a[(size_t)k * 4 + 3];
      const double s1 = a[(size_t)k * 4 + 0] + e1;
      const double s2 = a[(size_t)k * 4 + 1] + e2;
      const double mean = s1 / nt;
      const double var = nt > 1.0 ? (s2 - nt * mean * mean) / (nt - 1.0) : 0.0;
      const double qm = (E_eff / G.V_solid) * s1 * 1e-9;
      const double qs = (E_eff / G.V_solid) * 1e-9 * sqrt(fmax(var, 0.0) * nt);
      O.kn[((size_t)g * K + (k - 1)) * 2 + 0] = -qm / G.kappa_grad;
      O.kn[((size_t)g * K + (k - 1)) * 2 + 1] = qs / fabs(G.kappa_grad);
    }
  }
  if (O.q_bin && C.per_bin) {
    const double kb = E_eff / G.V_solid;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const size_t j = (size_t)g * n + i;
      double v = 0.0;
      if (C.f64_rep) {
        const size_t stride = (size_t)C.n_geoms * n;
#pragma unroll 8
        for (int r = 0; r < C.f64_rep; ++r) v += A.qbin[r * stride + j];
      } else {
        v = (double)A.qbinq[j] * kFxInv;
      }
      O.q_bin[j] = (kb * v) * 1e-9;
    }
  }
  if (threadIdx.x == 128) {   // (a warp the cells leave free)
    const double sx = A.dsc[g * 8 + 0], sx2 = A.dsc[g * 8 + 1];
    const double nt = (double)A.cnt[g * 4 + 3];
    const double mean = sx / nt;
    const double var = nt > 1.0 ? (sx2 - nt * mean * mean) / (nt - 1.0) : 0.0;
    const double q_mean = (E_eff / G.V_solid) * sx * 1e-9;
    const double q_se = (E_eff / G.V_solid) * 1e-9 * sqrt(fmax(var, 0.0) * nt);
    double* st = O.stats + (size_t)g * MCBTE_NSTATS;
    st[MCBTE_STAT_KAPPA] = -q_mean / G.kappa_grad;
    st[MCBTE_STAT_KAPPA_SE] = q_se / fabs(G.kappa_grad);
    st[MCBTE_STAT_Q_MEAN] = q_mean;
    st[MCBTE_STAT_Q_SE] = q_se;
    st[MCBTE_STAT_SUMX] = sx;
    st[MCBTE_STAT_SUMX2] = sx2;
    st[MCBTE_STAT_EVENTS] = (double)A.cnt[g * 4 + 0];
    st[MCBTE_STAT_TRUNCATED] = (double)A.cnt[g * 4 + 1];
    st[MCBTE_STAT_E_TOT] = G.E_tot;
    st[MCBTE_STAT_MAX_EVENTS] = (double)A.cnt[g * 4 + 2];
    st[MCBTE_STAT_KAPPA_CELL] = (-q_mean / G.kappa_grad) * (G.V_solid / G.V_box);
    st[MCBTE_STAT_SIGNED_EMITTED] = A.dsc[g * 8 + 2];
    st[MCBTE_STAT_SIGNED_ABSORBED] = A.dsc[g * 8 + 3];
    st[MCBTE_STAT_STATUS] = (flags[0] & 4)   ? (double)MCBTE_ERR_REPLAY
                            : (flags[0] & 1) ? (double)MCBTE_ERR_TIMEOUT
                                             : (A.cnt[g * 4 + 1] ? (double)MCBTE_WARN_TRUNCATED : 0.0);
    st[MCBTE_STAT_N] = nt;
    st[MCBTE_STAT_ABSORBED] = A.dsc[g * 8 + 7];
  }
  if (grad && g == 0) {
    // fold the copies of the gradient sums into the first
    double* gs = A.gsum;
    for (int i = threadIdx.x; i < kGradStride; i += blockDim.x) {
      double v = gs[i];
      for (int r = 1; r < kSumCopies; ++r) v += gs[(size_t)r * kGradStride + i];
      gs[i] = v;
    }
    __syncthreads();
    const double scale = -(E_eff / G.V_solid) * 1e-9 / G.kappa_grad;
    const double Rs = gs[0];
    for (int i = threadIdx.x; i < n; i += blockDim.x) O.dk[i] = scale * ((A.G[i] + (double)A.Gq[i] * kFxInv) + Rs * M.pi[i]);
    if (threadIdx.x == 0) {
      const double nt = (double)A.cnt[3];
      const double gm = gs[1] / nt;
      const double gv = (gs[2] - nt * gm * gm) / fmax(nt - 1.0, 1.0);
      const bool ok = G.pore && (C.mvd || (G.p_pore > 0.0 && G.p_pore < 1.0));
      const double nan = __longlong_as_double(0x7ff8000000000000ll);
      O.dkp[0] = ok ? scale * gs[1] : nan;
      O.dkp[1] = ok ? fabs(scale) * sqrt(fmax(gv, 0.0) * nt) : nan;
      for (int k = 0; k < C.n_dirs; ++k) {
        const double dm = gs[4 + 2 * k] / nt;
        const double dv = (gs[5 + 2 * k] - nt * dm * dm) / fmax(nt - 1.0, 1.0);
        O.dkdir[k * 2 + 0] = scale * gs[4 + 2 * k];
        O.dkdir[k * 2 + 1] = fabs(scale) * sqrt(fmax(dv, 0.0) * nt);
      }
    }
  }
}

__global__ void k_dirs_dot_pi(const double* dirs, int nd, MatView M, double* dpi) {
  const int k = threadIdx.x;
  if (k >= nd) return;
  double acc = 0.0;
  for (int i = 0; i < M.n; ++i) acc += dirs[(size_t)k * M.n + i] * M.pi[i];
  dpi[k] = acc;
}

template <bool CELLS, bool GRAD>
cudaError_t launch_f64(const GeoRun* geos, const uint64_t* offs, const MatView& M, const RunCfg& C, const Acc& A,
                       cudaStream_t s) {
  auto kern = k_steady_fp64<CELLS, GRAD>;
  const int blocks = f64_blocks(C.total);
  RunCfg R = C;
  R.take_chunk = take_chunk(C.total, (uint64_t)blocks * (kF64Threads / 32), 256u, (uint64_t)blocks * 4, 1u);
  kern<<<blocks, kF64Threads, 0, s>>>(geos, offs, M, R, A);
  return cudaGetLastError();
}
#endif  // MCBTE_F64

#if MCBTE_F32
// One persistent launch: SMs x resident blocks (or fewer on request).
template <int CELLS, bool GRAD, int TPB, bool EXT, int MODE>
cudaError_t launch_f32_kernel(const GeoRun* geos, const uint64_t* offs, const MatView& M, const RunCfg& C,
                              const Acc& A, int bps, cudaStream_t s) {
  // the gradient kernel keeps no cell tallies, and the per-bin flux only in
  // a fused pass
  const int nc = GRAD ? 0 : C.n_cells, pb = (GRAD && !C.fused) ? 0 : C.per_bin, snaps = (GRAD && C.mvd) ? TPB : 0;
  const SmemPlan S = MODE == 2 ? plan_tail(M.n, C.n_geoms, nc, pb, GRAD ? 1 : 0, snaps)
                               : plan_main(TPB, EXT, M.n, C.n_geoms, nc, pb, GRAD ? 1 : 0, snaps);
  auto kern = k_steady_f32<CELLS, GRAD, TPB, EXT, MODE>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S.bytes);
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, TPB, S.bytes);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaErrorInvalidConfiguration;
  const int b = (bps > 0 && bps < occ) ? bps : occ;
  RunCfg R = C;
  const uint64_t warps = (uint64_t)sm_count() * b * (TPB / 32);
  // a batch of geometries: about one chunk per warp, since a lane that comes
  // to another geometry flushes its sums (20 films of 180-9000 nm, 8e5
  // particles: 2.37 ms with four chunks per warp, 0.90 with one; 14e6 in 64
  // films 23.1 and 22.9)
  R.take_chunk = take_chunk(C.total, C.n_geoms > 1 ? (warps + 3) / 4 : warps, C.take_chunk, warps, 4u);
  kern<<<sm_count() * b, TPB, S.bytes, s>>>(geos, offs, M, R, A, S);
  return cudaGetLastError();
}

// Part 0: the main kernel alone.  Part 1: the main kernel that parks its
// tail, then the tail kernel over the parked particles (256-thread blocks).

template <int CELLS, bool GRAD, int TPB, bool EXT>
cudaError_t launch_f32_tpb(const GeoRun* geos, const uint64_t* offs, const MatView& M, const RunCfg& C,
                           const Acc& A, int bps, cudaStream_t s) {
#if MCBTE_F32_PART == 0
  return launch_f32_kernel<CELLS, GRAD, TPB, EXT, 0>(geos, offs, M, C, A, bps, s);
#else
  cudaError_t e = launch_f32_kernel<CELLS, GRAD, TPB, EXT, 1>(geos, offs, M, C, A, bps, s);
  if (e != cudaSuccess) return e;
  return launch_f32_kernel<CELLS, GRAD, kTailThreads, EXT, 2>(geos, offs, M, C, A, 0, s);
#endif
}

template <int CELLS, bool GRAD, bool EXT>
cudaError_t launch_f32_ext(const GeoRun* geos, const uint64_t* offs, const MatView& M, const RunCfg& C, const Acc& A,
                           int threads, int bps, cudaStream_t s) {
  switch (threads) {
    case 256: return launch_f32_tpb<CELLS, GRAD, 256, EXT>(geos, offs, M, C, A, bps, s);
    case 512: return launch_f32_tpb<CELLS, GRAD, 512, EXT>(geos, offs, M, C, A, bps, s);
    case 768: return launch_f32_tpb<CELLS, GRAD, 768, EXT>(geos, offs, M, C, A, bps, s);
    case 1024: return launch_f32_tpb<CELLS, GRAD, 1024, EXT>(geos, offs, M, C, A, bps, s);
    default: return cudaErrorInvalidValue;
  }
}

// The extended physics is compiled in only for runs that use it.
template <int CELLS, bool GRAD>
cudaError_t launch_f32(const GeoRun* geos, const uint64_t* offs, const MatView& M, const RunCfg& C, const Acc& A,
                       int threads, int bps, cudaStream_t s) {
  return C.ext ? launch_f32_ext<CELLS, GRAD, true>(geos, offs, M, C, A, threads, bps, s)
               : launch_f32_ext<CELLS, GRAD, false>(geos, offs, M, C, A, threads, bps, s);
}

cudaError_t launch_f32_variants(bool grad, bool cells, const GeoRun* geos, const uint64_t* offs, const MatView& M,
                                const RunCfg& C, const Acc& A, int threads, int bps, cudaStream_t s) {
  // the gradient pass keeps no cell or per-bin tallies
  if (grad) return launch_f32<0, true>(geos, offs, M, C, A, threads, bps, s);
  if (!cells) return launch_f32<0, false>(geos, offs, M, C, A, threads, bps, s);
  return C.cell_flux_axis ? launch_f32<2, false>(geos, offs, M, C, A, threads, bps, s)
                          : launch_f32<1, false>(geos, offs, M, C, A, threads, bps, s);
}
#endif  // MCBTE_F32

}  // namespace

#if MCBTE_F64
// SM count of the current device, cached per device ordinal (grids are sized
// for the device the launch goes to).
int sm_count() {
  constexpr int kDevices = 64;
  static std::atomic<int> cached[kDevices];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < kDevices) {
    const int c = cached[dev].load(std::memory_order_relaxed);
    if (c > 0) return c;
  }
  int v = 0;
  cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
  if (v < 1) v = 1;
  if (dev >= 0 && dev < kDevices) cached[dev].store(v, std::memory_order_relaxed);
  return v;
}

cudaError_t launch_steady(int precision, bool grad, const GeoRun* geos, const uint64_t* offs, const MatView& M,
                          const RunCfg& C, const Acc& A, int threads, int bps, cudaStream_t s) {
  const bool cells = C.n_cells > 0;
  if (precision == MCBTE_FP64_PLAIN) {
    if (grad) return cells ? launch_f64<true, true>(geos, offs, M, C, A, s) : launch_f64<false, true>(geos, offs, M, C, A, s);
    return cells ? launch_f64<true, false>(geos, offs, M, C, A, s) : launch_f64<false, false>(geos, offs, M, C, A, s);
  }
  // default block: 768 threads, 512 for the gradient (its estimator state
  // takes ~128 registers per thread)
  return launch_steady_f32(grad, cells, geos, offs, M, C, A, threads > 0 ? threads : (grad ? 512 : 768), bps, s);
}

cudaError_t launch_finalize_steady(const GeoRun* geos, const MatView& M, const RunCfg& C, const Acc& A,
                                   const SteadyOutDev& O, bool grad, const int* flags, cudaStream_t s) {
  k_finalize_steady<<<C.n_geoms, 256, 0, s>>>(geos, M, C, A, O, grad ? 1 : 0, flags);
  return cudaGetLastError();
}

cudaError_t launch_dirs_dot_pi(const double* dirs, int n_dirs, const MatView& M, double* dpi, cudaStream_t s) {
  if (n_dirs <= 0) return cudaSuccess;
  k_dirs_dot_pi<<<1, 32, 0, s>>>(dirs, n_dirs, M, dpi);
  return cudaGetLastError();
}
#endif  // MCBTE_F64

#if MCBTE_F32 && MCBTE_F32_PART == 1
cudaError_t launch_steady_f32_tail(bool grad, bool cells, const GeoRun* geos, const uint64_t* offs, const MatView& M,
                                   const RunCfg& C, const Acc& A, int threads, int bps, cudaStream_t s) {
  return launch_f32_variants(grad, cells, geos, offs, M, C, A, threads, bps, s);
}
#endif

#if MCBTE_F32 && MCBTE_F32_PART == 0
size_t park_record_bytes() { return (sizeof(ParkRec) + 15) & ~(size_t)15; }

// Runs that can park their tail (a park buffer and a threshold) take the
// kernels of part 1, the others the plain main kernel.
cudaError_t launch_steady_f32(bool grad, bool cells, const GeoRun* geos, const uint64_t* offs, const MatView& M,
                              const RunCfg& C, const Acc& A, int threads, int bps, cudaStream_t s) {
  if (A.park_cap > 0 && C.tail_max > 0)
    return launch_steady_f32_tail(grad, cells, geos, offs, M, C, A, threads, bps, s);
  return launch_f32_variants(grad, cells, geos, offs, M, C, A, threads, bps, s);
}
#endif  // MCBTE_F32

}  // namespace mcbte
