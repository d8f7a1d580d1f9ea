// Transient tracing (Secs. 3.2-3.5): wall sources emit at t0 = R t_max, the
// initial condition at t0 = 0 (Sec. 3.2); every measurement time inside a
// particle's life adds its snapshot to the detector grid (Eq. sampling).
// Persistent FP64 plain kernel and persistent FP32 kernel (per-lane refill,
// alias tables in shared memory, 64-bit fixed-point reductions into the
// [time][cell][T, qx, qy, qz] tally, which is far larger than shared memory).
#include "launch.h"

#ifndef MCBTE_F64
#define MCBTE_F64 0
#endif
#ifndef MCBTE_F32
#define MCBTE_F32 0
#endif

namespace mcbte {

namespace {

// First measurement index still ahead of the particle: for snapshots the
// first t_m >= t0, for bin averages the bin [t_{m-1}, t_m) containing t0.
__device__ __forceinline__ void transient_start(Particle<double>& p, const RunCfg& C) {
  int lo = 0, hi = C.n_times;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    const double tm = C.t_meas_ps[mid];
    if (C.time_average ? tm <= p.t : tm < p.t) lo = mid + 1; else hi = mid;
  }
  p.mi = lo;
}

// The run counters of a warp's finished particles, spread over its lanes:
// lane 0 events, 1 truncated, 2 most events, 3 traced, 4 sum of signs emitted,
// 5 sum of signs absorbed, 6 absorbed.  One register pair a lane, and one
// atomic per counter and warp at the kernel's end, where each particle added
// five to six to a few addresses (a wall pulse of 2e5 particles: 1.2e6
// atomics, two thirds of its kernel).
struct WarpAcct {
  unsigned long long v = 0ull;
  // called by all 32 lanes; `ended`: this lane's particle ended with `out`
  __device__ __forceinline__ void add(bool ended, int out, uint32_t e, float s, unsigned lane) {
    constexpr unsigned kAll = 0xffffffffu;
    const unsigned m = __ballot_sync(kAll, ended);
    if (!m) return;
    const unsigned mp = __ballot_sync(kAll, ended && s > 0.0f);
    const unsigned ma = __ballot_sync(kAll, ended && out == STEP_ABSORBED);
    const unsigned mt = __ballot_sync(kAll, ended && out == STEP_TRUNCATED);
    const unsigned nev = ended ? e + 1u : 0u;
    const unsigned lo = __reduce_add_sync(kAll, nev & 0xffffu), hi = __reduce_add_sync(kAll, nev >> 16);
    const unsigned mx = __reduce_max_sync(kAll, nev);
    const unsigned long long ev = ((unsigned long long)hi << 16) + lo;
    const long long se = 2ll * __popc(mp) - __popc(m), sa = 2ll * __popc(mp & ma) - __popc(ma);
    if (lane == 2) {
      v = mx > v ? mx : v;
    } else {
      v += lane == 0   ? ev
           : lane == 1 ? (unsigned long long)__popc(mt)
           : lane == 3 ? (unsigned long long)__popc(m)
           : lane == 4 ? (unsigned long long)se
           : lane == 5 ? (unsigned long long)sa
                       : (unsigned long long)__popc(ma);
    }
  }
  __device__ __forceinline__ void flush(unsigned lane, const Acc& A) const {
    unsigned long long* cnt = A.cnt + sum_copy() * 4;
    double* dsc = A.dsc + sum_copy() * 8;
    if (v == 0ull || lane > 6) return;
    if (lane == 2) atomicMax(cnt + 2, v);
    else if (lane < 4) atomicAdd(cnt + lane, v);
    else atomicAdd(dsc + (lane == 4 ? 2 : (lane == 5 ? 3 : 7)), (double)(long long)v);
  }
};

// The same in shared memory, added to by the lanes whose particles end.  For
// the FP32 kernel, whose steps are too short for WarpAcct's votes and whose
// threads have no registers for counters of their own (1e7 particles with the
// two-phonon clock: 116.1 ms with votes, 113.4 with a thread's counters in local
// memory, 110.5 here with the run of indices beside them).
struct SharedAcct {
  unsigned long long ev;
  unsigned traced, trunc, maxev, positive, absorbed, positive_absorbed;

  // by one lane of the warp
  __device__ __forceinline__ void reset() {
    ev = 0ull;
    traced = trunc = maxev = positive = absorbed = positive_absorbed = 0u;
  }
  __device__ __forceinline__ void end(int out, uint32_t e, float s) {
    const unsigned nev = e + 1u;
    atomicAdd(&ev, (unsigned long long)nev);
    atomicAdd(&traced, 1u);
    atomicMax(&maxev, nev);
    if (s > 0.0f) atomicAdd(&positive, 1u);
    if (out == STEP_TRUNCATED) atomicAdd(&trunc, 1u);
    if (out == STEP_ABSORBED) {
      atomicAdd(&absorbed, 1u);
      if (s > 0.0f) atomicAdd(&positive_absorbed, 1u);
    }
  }
  // called by all lanes of the warp
  __device__ __forceinline__ void flush(unsigned lane, const Acc& A) const {
    __syncwarp();
    if (lane != 0u || traced == 0u) return;
    unsigned long long* cnt = A.cnt + sum_copy() * 4;
    double* dsc = A.dsc + sum_copy() * 8;
    atomicAdd(cnt + 0, ev);
    if (trunc) atomicAdd(cnt + 1, (unsigned long long)trunc);
    atomicMax(cnt + 2, (unsigned long long)maxev);
    atomicAdd(cnt + 3, (unsigned long long)traced);
    atomicAdd(dsc + 2, (double)(2ll * positive - (long long)traced));
    if (absorbed) {
      atomicAdd(dsc + 3, (double)(2ll * positive_absorbed - (long long)absorbed));
      atomicAdd(dsc + 7, (double)absorbed);
    }
  }
};

// One finished particle added at once: bin averages, whose kernel has no
// register left for a lane's own counters (1e7 particles: 191.5 ms with them,
// 187.8 without) and whose particles are long.
__device__ __forceinline__ void transient_finish(const Particle<float>& p, int out, const Acc& A) {
  const unsigned long long nev = (unsigned long long)p.e + 1ull;
  unsigned long long* cnt = A.cnt + sum_copy() * 4;
  double* dsc = A.dsc + sum_copy() * 8;
  atomicAdd(cnt + 0, nev);
  if (out == STEP_TRUNCATED) atomicAdd(cnt + 1, 1ull);
  atomicMax(cnt + 2, nev);
  atomicAdd(cnt + 3, 1ull);
  atomicAdd(dsc + 2, (double)p.s);
  if (out == STEP_ABSORBED) {
    atomicAdd(dsc + 3, (double)p.s);
    atomicAdd(dsc + 7, 1.0);
  }
}

#if MCBTE_F64
// Persistent, like k_steady_fp64: 32 particles emitted at a time, a lane that
// is done refills.
__global__ void __launch_bounds__(kF64Threads, 1) k_transient_fp64(const GeoRun* __restrict__ geos, MatView M, RunCfg C,
                                                                   Acc A) {
  __shared__ Refill s_refill[kF64Threads / 32];
  __shared__ EmitBatch<double, true, true> s_batch[kF64Threads / 32];
  constexpr unsigned kAll = 0xffffffffu;
  const unsigned lane = threadIdx.x & 31u;
  const GeoRun& G = geos[0];
  const uint64_t deadline = *C.t0 + C.budget_ns;
  const uint2 key = run_key(C);
  Refill& refill = s_refill[threadIdx.x >> 5];
  EmitBatch<double, true, true>& batch = s_batch[threadIdx.x >> 5];
  refill.start(lane, C.take_chunk, C.total, deadline, A.flags);
  Particle<double> p;
  p.e = 0u;
  p.s = 0.0;
  WarpAcct acct;
  bool alive = false, pool_dry = false;
  for (;;) {
    const unsigned need = __ballot_sync(kAll, !alive);
    if (need && !pool_dry) {
      pool_dry = refill.hand_out(
          32, need, lane, A.work, C.total, deadline, A.flags,
          [&](uint64_t k) {
            emit_slot<double, true, true>(&batch, lane, geos, nullptr, 1, k, M, nullptr, key, C.t_max_ps);
          },
          [&](unsigned slot, uint64_t) {
            batch.load(slot, p, M, nullptr);
            transient_start(p, C);
            alive = true;
          });
    }
    if (!__any_sync(kAll, alive)) {
      if (pool_dry) break;
      continue;
    }
    int out = STEP_ALIVE;
    if (alive) {
      out = step_transient<double>(p, G, M, M.rec_relax, nullptr, C, key.x, key.y, A.snap, C.t_meas_ps, nullptr);
      if (out == STEP_ALIVE && (p.e & 1023u) == 0u && globaltimer_ns() > deadline) {
        atomicOr(A.flags, 1);
        out = STEP_TRUNCATED;
      }
    }
    const bool ended = alive && out != STEP_ALIVE;
    if (ended && A.events_pp) A.events_pp[p.pid] = p.e + 1u;
    acct.add(ended, out, p.e, (float)p.s, lane);
    if (ended) alive = false;
  }
  acct.flush(lane, A);
}

// Bin averages and detector regions: every lane traces one particle to its
// end, `share` particles a warp (32, fewer where a run has few).  What an event
// costs here is its walk through the detectors, which differs from lane to
// lane; with k_transient_fp64's vote after every event each waits for the
// longest walk of its warp (box of 64 x 64 x 32 cells, averages over 200 bins,
// 37 500 particles: 72.5 ms, 4.7 lanes active per instruction and 4.8e9 warp
// instructions; here 31.1, 7.5 and 2.9e9.  A quarter of that, 3750 particles:
// 16.0 and 14.4; snapshots into two regions, 150 000: 36.6 and 27.4).
__global__ void __launch_bounds__(kF64RegionThreads, 4) k_transient_fp64_regions(const GeoRun* __restrict__ geos,
                                                                                 MatView M, RunCfg C, Acc A,
                                                                                 unsigned share) {
  const unsigned lane = threadIdx.x & 31u;
  const uint64_t idx = ((uint64_t)blockIdx.x * (kF64RegionThreads / 32) + (threadIdx.x >> 5)) * share + lane;
  const GeoRun& G = geos[0];
  const uint64_t deadline = *C.t0 + C.budget_ns;
  const uint2 key = run_key(C);
  Particle<double> p;
  p.e = 0u;
  p.s = 0.0;
  int out = STEP_ALIVE;
  if (lane < share && idx < C.total) {
    if (globaltimer_ns() > deadline) {   // over budget before this particle started
      atomicOr(A.flags, 1);
    } else {
      p.pid = (uint32_t)idx;
      p.g = 0;
      emit<double>(p, G, M, M.rec_emit, M.rec_init, nullptr, key.x, key.y, true, C.t_max_ps);
      transient_start(p, C);
      for (;;) {
        out = step_transient<double>(p, G, M, M.rec_relax, nullptr, C, key.x, key.y, A.snap, C.t_meas_ps, nullptr);
        if (out != STEP_ALIVE) break;
        if ((p.e & 1023u) == 0u && globaltimer_ns() > deadline) {
          atomicOr(A.flags, 1);
          out = STEP_TRUNCATED;
          break;
        }
      }
      if (A.events_pp) A.events_pp[idx] = p.e + 1u;
    }
  }
  WarpAcct acct;
  acct.add(out != STEP_ALIVE, out, p.e, (float)p.s, lane);
  acct.flush(lane, A);
}

#endif  // MCBTE_F64
#if MCBTE_F32
// Particle state between time windows, 48 bytes: {x, t}, {u, d_rel},
// {event index, bin | sign bit, next measurement index | live bit, d2}
// (transient runs have no N_scat^max, so the relaxation count is not kept).
// Streaming (evict-first) accesses keep the window's tally slice in L2.
constexpr uint32_t kLive = 0x80000000u;

__device__ __forceinline__ void save_state(uint4* st, uint64_t idx, const Particle<float>& p) {
  uint4* q = st + idx * 3;
  __stcs(q + 0, make_uint4(__float_as_uint(p.x[0]), __float_as_uint(p.x[1]), __float_as_uint(p.x[2]),
                           __float_as_uint(p.t)));
  __stcs(q + 1, make_uint4(__float_as_uint(p.u[0]), __float_as_uint(p.u[1]), __float_as_uint(p.u[2]),
                           __float_as_uint(p.d_rel)));
  __stcs(q + 2, make_uint4(p.e, (uint32_t)p.bin | (p.s < 0.0f ? 0x80000000u : 0u), (uint32_t)p.mi | kLive,
                           __float_as_uint(p.d2)));
}

__device__ __forceinline__ void mark_done(uint4* st, uint64_t idx) { __stcs(st + idx * 3 + 2, make_uint4(0, 0, 0, 0)); }

// false: the particle ended in an earlier window, or it has nothing to
// sample before `win_end` (then its saved state stays as it is)
__device__ __forceinline__ bool load_state(const uint4* st, uint64_t idx, Particle<float>& p, const MatView& M,
                                           const float4* binf, const RunCfg& C) {
  const uint4* q = st + idx * 3;
  const uint4 c = __ldcs(q + 2);
  if (!(c.z & kLive)) return false;
  if (!C.win_last && (int)(c.z & ~kLive) >= C.win_end) return false;
  const uint4 a = __ldcs(q + 0);
  const uint4 b = __ldcs(q + 1);
  p.x[0] = __uint_as_float(a.x);
  p.x[1] = __uint_as_float(a.y);
  p.x[2] = __uint_as_float(a.z);
  p.t = __uint_as_float(a.w);
  p.u[0] = __uint_as_float(b.x);
  p.u[1] = __uint_as_float(b.y);
  p.u[2] = __uint_as_float(b.z);
  p.d_rel = __uint_as_float(b.w);
  p.e = c.x;
  p.bin = (int)(c.y & 0x7fffffffu);
  p.s = (c.y & 0x80000000u) ? -1.0f : 1.0f;
  p.mi = (int)(c.z & ~kLive);
  p.d2 = __uint_as_float(c.w);
  p.n_relax = 0;
  p.pid = (uint32_t)idx;
  p.g = 0;
  load_bin(p, M, binf);
  return true;
}

// Adds val[0..3] to the four words of tally record `rec` (kNoRec: nothing) of
// every lane.  The four lanes of a quad first transpose their values (two
// exchanges), so that each reduction instruction adds whole 32-byte records,
// the quad's lanes side by side: 8 sectors per instruction where a word per
// lane touched 32, four times each.  Called by all 32 lanes.  A tally has
// fewer than 2^32 - 1 records on the tracers' grids or `rec` is 64 bits wide.
constexpr unsigned kNoRec = 0xffffffffu;

template <typename Rec>
__device__ __forceinline__ void red_records(Rec rec, int val[4], double* snap, int lane) {
  constexpr unsigned kAll = 0xffffffffu;
  const bool b0 = (lane & 1) != 0, b1 = (lane & 2) != 0;
#pragma unroll
  for (int k = 0; k < 4; k += 2) {
    const int y = __shfl_xor_sync(kAll, b0 ? val[k] : val[k + 1], 1);
    if (b0) val[k] = y; else val[k + 1] = y;
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int y = __shfl_xor_sync(kAll, b1 ? val[k] : val[k + 2], 2);
    if (b1) val[k] = y; else val[k + 2] = y;
  }
  long long* q = reinterpret_cast<long long*>(snap) + (lane & 3);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const Rec rr = __shfl_sync(kAll, rec, (lane & ~3) | r);
    if (rr != (Rec)~(Rec)0) red_s64(q + (size_t)rr * 4, (long long)val[r]);
  }
}

// First index in [lo, n] whose measurement time is beyond t_end (closed: t_m <=
// t_end is not beyond).  Evenly spaced times, the usual request, are hit by
// the quotient t_end / spacing, checked against its two neighbours; any other
// case takes a bisection (eight dependent shared-memory reads for 200 times).
__device__ __forceinline__ int first_beyond(const float* tmeas, int lo, int n, float t_end, bool closed, float inv_dt) {
  const int g = min(max((int)(t_end * inv_dt), lo), n);
  auto covered = [&](int m) { return closed ? tmeas[m] <= t_end : tmeas[m] < t_end; };
  if ((g == n || !covered(g)) && (g == lo || covered(g - 1))) return g;
  int hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (covered(mid)) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// A warp's flights while their snapshots are shared out (shared memory).
struct FlightSlots {
  float4 xt[32];    // position and time at the flight's start
  float4 uv[32];    // direction, sign x speed
  int first[32];    // measurement index of the flight's first snapshot - its number in the warp
};

// Snapshots of a warp's flights, shared out over its 32 lanes.  Lane i
// takes k_i snapshots this step (measurement indices p.mi .. p.mi + k_i - 1
// of the flight that starts at p.x at time p.t); a lane's count depends on
// its flight's length, so a per-lane loop would leave most lanes idle while
// the longest flights sample.  Here the warp's k_1 + ... + k_32 snapshots are
// taken 32 at a time.  Every lane of the warp must call this (k = 0 for idle
// lanes).  The arithmetic per snapshot is the per-lane loop's (Eq. sampling,
// Sec. 3.4).
//
// Whole records (C.snap_records: 2 always, 1 where the step has 24 snapshots
// or more): the flights that have snapshots are written to `fs`, side by side in
// lane order; where each begins among the 32 of a round is one bit of a mask,
// so a lane finds its snapshot's flight by a population count, and the quads
// add their records (red_records).  Fewer reductions, more instructions.
// Word by word: a bisection of the prefix sums and shuffles of the owner's
// state, four reductions per lane.  transient_snap_records() chooses.
__device__ __forceinline__ void warp_snapshots(int k, const Particle<float>& p, const float* tmeas, const float* cinv,
                                               const RunCfg& C, double* snap, FlightSlots& fs) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = (int)(threadIdx.x & 31u);
  const unsigned some = __ballot_sync(kAll, k > 0);
  if (!some) return;
  int incl = k;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kAll, incl, o);
    if (lane >= o) incl += y;
  }
  const int total = __shfl_sync(kAll, incl, 31);
  const int nx = C.grid[0], ny = C.grid[1], nz = C.grid[2];
  const size_t ncell = (size_t)nx * ny * nz;
  if (C.snap_records == 0 || (C.snap_records == 1 && total < 24)) {
    for (int base = 0; base < total; base += 32) {
      const int j = base + lane;
      // owner: the first lane whose inclusive sum exceeds j (always in 0..31)
      int own = 0;
#pragma unroll
      for (int st = 16; st >= 1; st >>= 1) {
        const int v = __shfl_sync(kAll, incl, own + st - 1);
        if (v <= j) own += st;
      }
      const int first = __shfl_sync(kAll, incl - k, own);
      const int mi0 = __shfl_sync(kAll, p.mi, own);
      const float x0 = __shfl_sync(kAll, p.x[0], own), x1 = __shfl_sync(kAll, p.x[1], own),
                  x2 = __shfl_sync(kAll, p.x[2], own);
      const float u0 = __shfl_sync(kAll, p.u[0], own), u1 = __shfl_sync(kAll, p.u[1], own),
                  u2 = __shfl_sync(kAll, p.u[2], own);
      const float t0 = __shfl_sync(kAll, p.t, own), v = __shfl_sync(kAll, p.v, own), s = __shfl_sync(kAll, p.s, own);
      if (j < total) {
        const int m = mi0 + (j - first);
        const float dist = v * (tmeas[m] - t0);
        const float pm0 = x0 + dist * u0, pm1 = x1 + dist * u1, pm2 = x2 + dist * u2;
        const int ix = min(max((int)floorf(pm0 * cinv[0]), 0), nx - 1);
        const int iy = min(max((int)floorf(pm1 * cinv[1]), 0), ny - 1);
        const int iz = min(max((int)floorf(pm2 * cinv[2]), 0), nz - 1);
        long long* q = reinterpret_cast<long long*>(snap) + ((size_t)m * ncell + ((size_t)iz * ny + iy) * nx + ix) * 4;
        const float sv = s * v;
        red_s64(q + 0, s > 0.0f ? 1ll : -1ll);
        if (v < 1024.0f) {
          // |s v u_a| <= v (1 + rounding): below 2^30 in fixed point, so the
          // 32-bit conversion gives the value fx gives
          red_s64(q + 1, (long long)__float2int_rn((sv * u0) * kFx));
          red_s64(q + 2, (long long)__float2int_rn((sv * u1) * kFx));
          red_s64(q + 3, (long long)__float2int_rn((sv * u2) * kFx));
        } else {
          red_s64(q + 1, fx(sv * u0));
          red_s64(q + 2, fx(sv * u1));
          red_s64(q + 3, fx(sv * u2));
        }
      }
    }
    return;
  }
  const int excl = incl - k;
  if (k > 0) {
    const int r = __popc(some & ((1u << lane) - 1u));
    fs.xt[r] = make_float4(p.x[0], p.x[1], p.x[2], p.t);
    fs.uv[r] = make_float4(p.u[0], p.u[1], p.u[2], p.s * p.v);
    fs.first[r] = p.mi - excl;
  }
  __syncwarp();
  const bool narrow = ncell * (size_t)C.n_times < (size_t)kNoRec;
  int before = -1;   // flights that begin before this round, less one
  for (int base = 0; base < total; base += 32) {
    const int rel = excl - base;
    const unsigned begins = __reduce_or_sync(kAll, (k > 0 && rel >= 0 && rel < 32) ? 1u << rel : 0u);
    const int j = base + lane;
    unsigned long long rec = ~0ull;
    int val[4] = {0, 0, 0, 0};
    if (j < total) {
      const int f = before + __popc(begins & (0xffffffffu >> (31 - lane)));
      const float4 xt = fs.xt[f], uv = fs.uv[f];
      const int m = fs.first[f] + j;
      const float sv = uv.w, v = fabsf(sv);
      const float dist = v * (tmeas[m] - xt.w);
      const float pm0 = xt.x + dist * uv.x, pm1 = xt.y + dist * uv.y, pm2 = xt.z + dist * uv.z;
      const int ix = min(max((int)floorf(pm0 * cinv[0]), 0), nx - 1);
      const int iy = min(max((int)floorf(pm1 * cinv[1]), 0), ny - 1);
      const int iz = min(max((int)floorf(pm2 * cinv[2]), 0), nz - 1);
      rec = narrow ? (unsigned long long)(((unsigned)m * (unsigned)nz + (unsigned)iz) * (unsigned)ny + (unsigned)iy) * nx + ix
                   : (unsigned long long)m * ncell + ((size_t)iz * ny + iy) * nx + ix;
      if (v < 1024.0f) {
        // |s v u_a| <= v (1 + rounding): below 2^30 in fixed point, so the
        // 32-bit conversion gives the value fx gives
        val[0] = sv > 0.0f ? 1 : -1;
        val[1] = __float2int_rn((sv * uv.x) * kFx);
        val[2] = __float2int_rn((sv * uv.y) * kFx);
        val[3] = __float2int_rn((sv * uv.z) * kFx);
      } else {
        // beyond 32 bits in fixed point: this lane adds its own record
        long long* q = reinterpret_cast<long long*>(snap) + rec * 4;
        red_s64(q + 0, sv > 0.0f ? 1ll : -1ll);
        red_s64(q + 1, fx(sv * uv.x));
        red_s64(q + 2, fx(sv * uv.y));
        red_s64(q + 3, fx(sv * uv.z));
        rec = ~0ull;
      }
    }
    before += __popc(begins);
    if (narrow) red_records<unsigned>((unsigned)rec, val, snap, lane);
    else red_records<unsigned long long>(rec, val, snap, lane);
  }
  __syncwarp();   // the slots are rewritten at the next step
}

// Time-bin averages of a warp's flights, shared out over its 32 lanes in the
// same way: lane i contributes to the k_i bins m = p.mi .. p.mi + k_i - 1
// that its flight [p.t, t_end) overlaps; each (flight, bin) pair is one item,
// and the warp takes its items 32 at a time, every lane walking its item's
// piece of flight through the detector grids (region_track) with the
// owner's state read by shuffles.  Every lane of the warp must call this.
// The arithmetic per item is the per-lane loop's in step_transient.
__device__ __forceinline__ void warp_bin_averages(int k, float t_end, const Particle<float>& p, const float* tmeas,
                                                  const RunCfg& C, double* snap) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = (int)(threadIdx.x & 31u);
  int incl = k;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kAll, incl, o);
    if (lane >= o) incl += y;
  }
  const int total = __shfl_sync(kAll, incl, 31);
  for (int base = 0; base < total; base += 32) {
    const int j = base + lane;
    int own = 0;
#pragma unroll
    for (int st = 16; st >= 1; st >>= 1) {
      const int v = __shfl_sync(kAll, incl, own + st - 1);
      if (v <= j) own += st;
    }
    const int first = __shfl_sync(kAll, incl - k, own);
    const int mi0 = __shfl_sync(kAll, p.mi, own);
    const float x[3] = {__shfl_sync(kAll, p.x[0], own), __shfl_sync(kAll, p.x[1], own),
                        __shfl_sync(kAll, p.x[2], own)};
    const float u0 = __shfl_sync(kAll, p.u[0], own), u1 = __shfl_sync(kAll, p.u[1], own),
                u2 = __shfl_sync(kAll, p.u[2], own);
    const float t0 = __shfl_sync(kAll, p.t, own), te = __shfl_sync(kAll, t_end, own),
                v = __shfl_sync(kAll, p.v, own), s = __shfl_sync(kAll, p.s, own);
    if (j < total) {
      const int m = mi0 + (j - first);
      const float b0 = m == 0 ? 0.0f : tmeas[m - 1];
      const float b1 = tmeas[m];
      const float ta = t0 > b0 ? t0 : b0;
      const float tb = te < b1 ? te : b1;
      if (ta < tb) {
        const float wb = 1.0f / (b1 - b0);
        const float w3[3] = {v * u0, v * u1, v * u2};
        for (int r = 0; r < C.n_regs; ++r) {
          const DetRegion& reg = C.regs[r];
          const size_t base_c = (size_t)m * C.n_det + reg.off;
          region_track<float>(reg, x, w3, t0, ta, tb, [&](uint32_t det, float dur) {
            long long* q = reinterpret_cast<long long*>(snap) + (base_c + det) * 4;
            const float f = (s * dur) * wb;
            red_s64(q + 0, fx(f));
            red_s64(q + 1, fx((f * v) * u0));
            red_s64(q + 2, fx((f * v) * u1));
            red_s64(q + 3, fx((f * v) * u2));
          });
        }
      }
    }
  }
}

// Shared memory: the warps' flight slots (snapshots), the measurement times as
// float (always), then the relaxation alias records and per-bin constants where
// the plan has room.
// TAVG: the run tallies time-bin averages (compiled apart, so that the
// snapshot variant carries none of that code).
template <int TPB, bool EXT, bool TAVG>
__global__ void __launch_bounds__(TPB, 1) k_transient_f32(const GeoRun* __restrict__ geos, MatView M, RunCfg C,
                                                          Acc A, SmemPlan S) {
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned char* sp = smem;
  const int n = M.n;
  const uint4* relax = M.rec_relax;
  const float4* binf = M.binf;
  // the warps' flight slots first (16-byte aligned), then the measurement times
  FlightSlots* slots = nullptr;
  if constexpr (!TAVG) {
    slots = reinterpret_cast<FlightSlots*>(sp) + (threadIdx.x >> 5);
    sp += (TPB / 32) * sizeof(FlightSlots);
  }
  float* tmeas = reinterpret_cast<float*>(sp);
  for (int i = threadIdx.x; i < C.n_times; i += TPB) tmeas[i] = (float)C.t_meas_ps[i];
  sp += ((size_t)C.n_times * sizeof(float) + 15) & ~(size_t)15;
  if (S.relax_in_smem) {
    uint4* t = reinterpret_cast<uint4*>(sp);
    for (int i = threadIdx.x; i < n; i += TPB) t[i] = M.rec_relax[i];
    relax = t;
    sp += (size_t)n * sizeof(uint4);
  }
  if (S.binf_in_smem) {
    float4* t = reinterpret_cast<float4*>(sp);
    for (int i = threadIdx.x; i < n; i += TPB) t[i] = M.binf[i];
    binf = t;
  }
  __syncthreads();
  const GeoRun& G = geos[0];
  float cinv[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) cinv[a] = (float)((double)C.grid[a] / G.L[a]);
  const float inv_dt = (float)C.n_times / tmeas[C.n_times - 1];
  const uint64_t deadline = *C.t0 + C.budget_ns;
  const unsigned lane = threadIdx.x & 31u;
  const uint2 key = run_key(C);
  // the warp's particle indices not yet handed out
  __shared__ WarpRun s_run[TPB / 32];
  {
    WarpRun r;
    r.start(C.take_chunk, C.total, deadline, A.flags);
    if (lane == 0) s_run[threadIdx.x >> 5] = r;
    __syncwarp();
  }
  auto take = [&](unsigned need) -> uint64_t {
    WarpRun r = s_run[threadIdx.x >> 5];
    __syncwarp();
    const uint64_t k = r.take(need, lane, A.work, C.total, deadline, A.flags);
    if (lane == 0) s_run[threadIdx.x >> 5] = r;
    __syncwarp();
    return k;
  };
  Particle<float> p;
  p.e = 0u;
  p.s = 0.0f;
  __shared__ SharedAcct s_acct[TAVG ? 1 : TPB / 32];
  SharedAcct& acct = s_acct[TAVG ? 0 : threadIdx.x >> 5];
  if (!TAVG && lane == 0u) acct.reset();
  __syncwarp();
  bool alive = false;
  bool drained = false;   // as in the steady tracer: idle lanes stay until the warp is drained
  uint64_t idx = 0;
  constexpr unsigned kAll = 0xffffffffu;
  if (TAVG || C.n_regs == 0) {
    // Snapshots on the whole-box grid: every lane of a warp runs every step
    // (no lane skips ahead to the next refill), so that the warp can share
    // out its snapshots (warp_snapshots).  Flight and event as in
    // step_transient.
    for (;;) {
      if (__all_sync(kAll, drained)) break;
      const unsigned need = __ballot_sync(kAll, !alive && !drained);
      if (need) {
        const uint64_t k = take(need);
        if (!alive && !drained) {
          idx = k;
          if (idx >= C.total || (*(volatile int*)A.flags & 1)) {
            drained = true;
          } else if (C.win_first) {
            p.pid = (uint32_t)idx;
            p.g = 0;
            emit<float, EXT>(p, G, M, M.rec_emit, M.rec_init, binf, key.x, key.y, true, (float)C.t_max_ps);
            p.mi = first_beyond(tmeas, 0, C.n_times, p.t, TAVG, inv_dt);   // (bins: the one that holds the emission)
            if (!C.win_last && p.mi >= C.win_end) save_state(A.tstate, idx, p);   // emitted after this window
            else alive = true;
          } else if (load_state(A.tstate, idx, p, M, binf, C)) {
            alive = true;
          }
        }
      }
      // the flight: nearest of t_max, the clocks and the boundary (Sec. 3.3,
      // Sec. 3.5.6), and how many measurement times it covers
      int out = STEP_ALIVE, k = 0, face = 0, mi_next = 0;
      bool fin = false, rlx = false, rlx2 = false;
      float seg = 0.0f, t_end = 0.0f;
      if (alive) {
        if (p.e + 1u >= C.max_events) {
          out = STEP_TRUNCATED;
        } else {
          float db;
          first_hit<float, EXT>(G, p.x, p.u, p.d_rel, &db, &face);
          const float tmax = (float)C.t_max_ps;
          const float d_end = (tmax - p.t) * p.v;
          if (d_end <= p.d_rel && d_end <= db && (!EXT || d_end <= p.d2)) { fin = true; seg = d_end; }
          else if (p.d_rel < db && (!EXT || p.d_rel <= p.d2)) { rlx = true; seg = p.d_rel; }
          else if (EXT && p.d2 < db) { rlx2 = true; seg = p.d2; }
          else { seg = db; }
          t_end = fin ? tmax : p.t + seg * p.inv_v;
          if constexpr (TAVG) {
            // the bins [t_{m-1}, t_m) the flight overlaps: m = p.mi up to the
            // first m whose end t_m lies beyond t_end (the flight's last bin,
            // where the particle stays)
            mi_next = first_beyond(tmeas, p.mi, C.n_times, t_end, true, inv_dt);
            k = p.mi < C.n_times ? (mi_next < C.n_times ? mi_next : C.n_times - 1) - p.mi + 1 : 0;
          } else {
            // the measurement times in [t, t_end) (closed at t_max)
            k = first_beyond(tmeas, p.mi, C.n_times, t_end, fin, inv_dt) - p.mi;
          }
        }
      }
      if constexpr (TAVG) warp_bin_averages(k, t_end, p, tmeas, C, A.snap);
      else warp_snapshots(k, p, tmeas, cinv, C, A.snap, *slots);
      if (alive) {
        if (out == STEP_ALIVE) {
          if constexpr (TAVG) p.mi = mi_next;
          else p.mi += k;
          p.t = t_end;
#pragma unroll
          for (int a = 0; a < 3; ++a) p.x[a] = p.x[a] + seg * p.u[a];
          if (fin) {
            out = STEP_DONE;
          } else {
            GradOff off;
            out = apply_event<float, GradOff, TallyNone, EXT>(p, G, M, relax, binf, C, key.x, key.y, rlx, rlx2, face, seg,
                                                              TallyNone(), off, 0.0);
          }
        }
        if (out == STEP_ALIVE && (p.e & 255u) == 0u && globaltimer_ns() > deadline) {
          atomicOr(A.flags, 1);
          out = STEP_TRUNCATED;
        }
        if (out != STEP_ALIVE) {
          if constexpr (TAVG) transient_finish(p, out, A);
          else acct.end(out, p.e, p.s);
          alive = false;
          if (A.events_pp) A.events_pp[idx] = p.e + 1u;
          if (!C.win_last) mark_done(A.tstate, idx);
        } else if (!C.win_last && p.mi >= C.win_end) {
          save_state(A.tstate, idx, p);
          alive = false;
        }
      }
    }
    if constexpr (!TAVG) acct.flush(lane, A);
    return;
  }
  // snapshots into detector regions: the per-lane loop
  if constexpr (!TAVG) {
    for (;;) {
      if (__all_sync(kAll, drained)) break;
      const unsigned need = __ballot_sync(kAll, !alive && !drained);
      if (need) {
        const uint64_t k = take(need);
        if (!alive && !drained) {
          idx = k;
          if (idx >= C.total || (*(volatile int*)A.flags & 1)) {
            drained = true;
          } else if (C.win_first) {
            p.pid = (uint32_t)idx;
            p.g = 0;
            emit<float, EXT>(p, G, M, M.rec_emit, M.rec_init, binf, key.x, key.y, true, (float)C.t_max_ps);
            p.mi = first_beyond(tmeas, 0, C.n_times, p.t, TAVG, inv_dt);   // (bins: the one that holds the emission)
            if (!C.win_last && p.mi >= C.win_end) save_state(A.tstate, idx, p);   // emitted after this window
            else alive = true;
          } else if (load_state(A.tstate, idx, p, M, binf, C)) {
            alive = true;
          }
        }
      }
      int out = STEP_ALIVE;
      if (alive) {
        out = step_transient<float, EXT>(p, G, M, relax, binf, C, key.x, key.y, A.snap, tmeas, cinv);
        if (out == STEP_ALIVE && (p.e & 255u) == 0u && globaltimer_ns() > deadline) {
          atomicOr(A.flags, 1);
          out = STEP_TRUNCATED;
        }
        if (out != STEP_ALIVE) {
          acct.end(out, p.e, p.s);
          alive = false;
          if (A.events_pp) A.events_pp[idx] = p.e + 1u;
          if (!C.win_last) mark_done(A.tstate, idx);
        } else if (!C.win_last && p.mi >= C.win_end) {
          // this window's snapshots are taken: park the particle at its event
          save_state(A.tstate, idx, p);
          alive = false;
        }
      }
    }
    acct.flush(lane, A);
  }
}

#endif  // MCBTE_F32
#if MCBTE_F64
// q as a double, exactly: for |q| < 2^53 the bits are put together by integer
// instructions (a conversion takes the FP64 pipe, the finaliser's bottleneck).
__device__ __forceinline__ double exact_double(long long q) {
  const unsigned long long m = q < 0 ? 0ull - (unsigned long long)q : (unsigned long long)q;
  if (m == 0ull) return 0.0;
  if (m >> 53) return (double)q;
  const int z = __clzll((long long)m);   // 11..63
  const unsigned long long bits =
      ((unsigned long long)(1086 - z) << 52) | ((m << (z - 11)) & 0x000fffffffffffffull);
  return __longlong_as_double((long long)(bits | ((unsigned long long)q & 0x8000000000000000ull)));
}

// Scale the raw snapshot sums: T = s E_eff / (C V_cell), q = s E_eff V_g / V_cell.
// `fixed`: the sums are the FP32 path's integers (signed count; flux in
// 2^-20 nm/ps units), converted here in place.
__global__ void k_finalize_transient(const GeoRun* geos, MatView M, RunCfg C, Acc A, double* tally, double* stats,
                                     size_t n_cells_total, int fixed) {
  const GeoRun& G = geos[0];
  const double E_eff = G.E_tot / (double)G.n;
  const double Vc = G.V_box / (double)((size_t)C.grid[0] * C.grid[1] * C.grid[2]);
  const size_t total = (size_t)C.n_times * n_cells_total;
  // (16-byte loads and stores: a caller's tally may be aligned to 8 only)
  const bool wide = ((reinterpret_cast<uintptr_t>(A.snap) | reinterpret_cast<uintptr_t>(tally)) & 15u) == 0;
  if (fixed && C.n_regs == 0 && !C.time_average && wide) {
    // Snapshots on the whole-box grid: one pass over the tally, bound by its
    // 64 bytes of traffic per entry once the FP64 work is four products and no
    // quotient (the factors are the same for every entry; the FP64 pipe takes
    // 1/64 of the FP32 rate).
    const double kT = E_eff / (M.sums[0] * Vc);
    const double kq = ((E_eff / Vc) * kFxInv) * 1e3;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
      const longlong2* r = reinterpret_cast<const longlong2*>(A.snap + i * 4);
      double2* o = reinterpret_cast<double2*>(tally + i * 4);
      const longlong2 q0 = r[0], q1 = r[1];
      o[0] = make_double2(kT * exact_double(q0.x), kq * exact_double(q0.y));
      o[1] = make_double2(kq * exact_double(q1.x), kq * exact_double(q1.y));
    }
  } else {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
      // volume of this entry's detector (its region's split, or the grid cell)
      double vd = Vc;
      if (C.n_regs > 0) {
        const uint32_t det = (uint32_t)(i % n_cells_total);
        for (int k = 0; k < C.n_regs; ++k)
          if (det >= C.regs[k].off) vd = C.regs[k].v_det;
      }
      const double kT = E_eff / (M.sums[0] * vd);
      const double kq = E_eff / vd;
      const double* r = A.snap + i * 4;
      double* o = tally + i * 4;
      double a0, a1, a2, a3;
      if (fixed) {
        const long long* q = reinterpret_cast<const long long*>(r);
        a0 = C.time_average ? (double)q[0] * kFxInv : (double)q[0];
        a1 = (double)q[1] * kFxInv;
        a2 = (double)q[2] * kFxInv;
        a3 = (double)q[3] * kFxInv;
      } else {
        a0 = r[0];
        a1 = r[1];
        a2 = r[2];
        a3 = r[3];
      }
      o[0] = kT * a0;
      o[1] = (kq * a1) * 1e3;
      o[2] = (kq * a2) * 1e3;
      o[3] = (kq * a3) * 1e3;
    }
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x < 32) {
    // fold the copies of the run counters: a lane per copy, then a warp sum
    // (whole numbers, so the order changes nothing)
    const unsigned lane = threadIdx.x;
    unsigned long long c[4] = {0ull, 0ull, 0ull, 0ull};
    double d[3] = {0.0, 0.0, 0.0};
    for (int r = (int)lane; r < kSumCopies; r += 32) {
      c[0] += A.cnt[r * 4 + 0];
      c[1] += A.cnt[r * 4 + 1];
      c[2] = c[2] > A.cnt[r * 4 + 2] ? c[2] : A.cnt[r * 4 + 2];
      c[3] += A.cnt[r * 4 + 3];
      d[0] += A.dsc[r * 8 + 2];
      d[1] += A.dsc[r * 8 + 3];
      d[2] += A.dsc[r * 8 + 7];
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      c[0] += __shfl_xor_sync(0xffffffffu, c[0], o);
      c[1] += __shfl_xor_sync(0xffffffffu, c[1], o);
      const unsigned long long m = __shfl_xor_sync(0xffffffffu, c[2], o);
      c[2] = c[2] > m ? c[2] : m;
      c[3] += __shfl_xor_sync(0xffffffffu, c[3], o);
      for (int k = 0; k < 3; ++k) d[k] += __shfl_xor_sync(0xffffffffu, d[k], o);
    }
    if (lane == 0) {
      for (int k = 0; k < MCBTE_NSTATS; ++k) stats[k] = 0.0;
      stats[MCBTE_STAT_EVENTS] = (double)c[0];
      stats[MCBTE_STAT_TRUNCATED] = (double)c[1];
      stats[MCBTE_STAT_MAX_EVENTS] = (double)c[2];
      stats[MCBTE_STAT_N] = (double)c[3];
      stats[MCBTE_STAT_E_TOT] = G.E_tot;
      stats[MCBTE_STAT_SIGNED_EMITTED] = d[0];
      stats[MCBTE_STAT_SIGNED_ABSORBED] = d[1];
      stats[MCBTE_STAT_ABSORBED] = d[2];
      stats[MCBTE_STAT_STATUS] = (A.flags[0] & 1) ? (double)MCBTE_ERR_TIMEOUT
                                                  : (c[1] ? (double)MCBTE_WARN_TRUNCATED : 0.0);
    }
  }
}

#endif  // MCBTE_F64
}  // namespace

#if MCBTE_F64
cudaError_t launch_transient(int precision, const GeoRun* geos, const MatView& M, const RunCfg& C, const Acc& A,
                             int threads, int bps, cudaStream_t s) {
  if (precision == MCBTE_FP64_PLAIN && C.n_regs > 0) {
    // a warp on every scheduler first, as in take_chunk
    const uint64_t spread = (uint64_t)sm_count() * 4;
    const uint64_t share = C.total > 32 * spread ? 32 : (C.total + spread - 1) / spread;
    const uint64_t per_block = share * (kF64RegionThreads / 32);
    k_transient_fp64_regions<<<(unsigned)((C.total + per_block - 1) / per_block), kF64RegionThreads, 0, s>>>(
        geos, M, C, A, (unsigned)share);
    return cudaGetLastError();
  }
  if (precision == MCBTE_FP64_PLAIN) {
    const int blocks = f64_blocks(C.total);
    RunCfg R = C;
    R.take_chunk = take_chunk(C.total, (uint64_t)blocks * (kF64Threads / 32), 256u, (uint64_t)blocks * 4, 1u);
    k_transient_fp64<<<blocks, kF64Threads, 0, s>>>(geos, M, R, A);
    return cudaGetLastError();
  }
  return launch_transient_f32(geos, M, C, A, threads > 0 ? threads : 1024, bps, s);
}

#endif  // MCBTE_F64
#if MCBTE_F32
namespace {
template <int TPB, bool EXT, bool TAVG>
cudaError_t launch_transient_tav(const GeoRun* geos, const MatView& M, const RunCfg& C, const Acc& A, int bps,
                                 cudaStream_t s) {
  const size_t tm_bytes = (((size_t)C.n_times * sizeof(float) + 15) & ~(size_t)15) +
                          (TAVG ? 0 : (TPB / 32) * sizeof(FlightSlots));
  SmemPlan S = plan_tables(M.n, 1, 0, 0, 200 * 1024 - tm_bytes);
  S.bytes += tm_bytes;
  auto kern = k_transient_f32<TPB, EXT, TAVG>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S.bytes);
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, TPB, S.bytes);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaErrorInvalidConfiguration;
  const int b = (bps > 0 && bps < occ) ? bps : occ;
  RunCfg R = C;
  const uint64_t warps = (uint64_t)sm_count() * b * (TPB / 32);
  R.take_chunk = take_chunk(C.total, warps, C.take_chunk, warps, 4u);
  kern<<<sm_count() * b, TPB, S.bytes, s>>>(geos, M, R, A, S);
  return cudaGetLastError();
}
template <int TPB, bool EXT>
cudaError_t launch_transient_tpb(const GeoRun* geos, const MatView& M, const RunCfg& C, const Acc& A, int bps,
                                 cudaStream_t s) {
  return C.time_average ? launch_transient_tav<TPB, EXT, true>(geos, M, C, A, bps, s)
                        : launch_transient_tav<TPB, EXT, false>(geos, M, C, A, bps, s);
}
}  // namespace

cudaError_t launch_transient_f32(const GeoRun* geos, const MatView& M, const RunCfg& C, const Acc& A, int threads,
                                 int bps, cudaStream_t s) {
  const bool imp = C.ext != 0;   // the extended physics is compiled in only when used
  switch (threads) {
    case 256: return imp ? launch_transient_tpb<256, true>(geos, M, C, A, bps, s)
                         : launch_transient_tpb<256, false>(geos, M, C, A, bps, s);
    case 512: return imp ? launch_transient_tpb<512, true>(geos, M, C, A, bps, s)
                         : launch_transient_tpb<512, false>(geos, M, C, A, bps, s);
    case 768: return imp ? launch_transient_tpb<768, true>(geos, M, C, A, bps, s)
                         : launch_transient_tpb<768, false>(geos, M, C, A, bps, s);
    case 1024: return imp ? launch_transient_tpb<1024, true>(geos, M, C, A, bps, s)
                          : launch_transient_tpb<1024, false>(geos, M, C, A, bps, s);
    default: return cudaErrorInvalidValue;
  }
}

#endif  // MCBTE_F32
#if MCBTE_F64
cudaError_t launch_finalize_transient(const GeoRun* geos, const MatView& M, const RunCfg& C, const Acc& A,
                                      double* tally, double* stats, size_t n_cells_total, bool fixed,
                                      cudaStream_t s) {
  k_finalize_transient<<<sm_count() * 4, 256, 0, s>>>(geos, M, C, A, tally, stats, n_cells_total, fixed ? 1 : 0);
  return cudaGetLastError();
}

#endif  // MCBTE_F64

}  // namespace mcbte
