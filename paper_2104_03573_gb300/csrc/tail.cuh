// The FP32 steady tracer's tail: the event loops of the tail kernel, for warps
// whose last particles run on alone.  Such a run's length is its longest
// particle's chain of dependent events, so these loops are laid out for
// latency: everything an event draws is computed ahead on all lanes
// (DrawLean), quantities of a direction (reciprocals, target faces) are kept
// from event to event, and the event itself holds the geometry only.  Every
// value is the event step's own (step_steady, apply_event) bit for bit.
// Cycles per event of a lone particle (gray, 1 mm free path; 2.07 GHz), before
// and now: 10 nm film 518 -> 197 (half specular walls 518 -> 198, specular 501 ->
// 200), pore lattice 771 -> 452, its measure-valued gradient 1470 -> 828 and
// likelihood-ratio gradient 999 -> 470, square-pore mesh 1374 -> 767.
#pragma once

#include "tracer.cuh"

namespace mcbte {

// What an event's random words decide, and what follows from them alone: the
// draws of Draw32, the reciprocals of both directions' components (0 where a
// component is 0), the relaxation's new distance, and the specular test
// against every surface of the geometry (bits 0-5 faces, 6 the pore, 7 + k
// wall k).  80 bytes, so that a gradient's slots leave room for its pore-hit
// snapshots; a film (trace_film) needs no reciprocals and keeps in their place
// {lam[1], lam[2], lam[0], the length of the flight across} and {its tally from
// the lower wall (64 bits), the relaxation's distance}.
struct __align__(16) DrawLean : Draw32 {
  float riso[3];
  float d_new;
  float rlam[3];
  uint32_t spec;

  __device__ __forceinline__ float4 film_flight() const { return make_float4(riso[0], riso[1], riso[2], d_new); }
  __device__ __forceinline__ long long film_tally() const {
    return (long long)(((unsigned long long)__float_as_uint(rlam[1]) << 32) | __float_as_uint(rlam[0]));
  }
  __device__ __forceinline__ float film_d_new() const { return rlam[2]; }
  // W: the film's wall axis; s: the particle's sign
  __device__ __forceinline__ void to_film(float LW, int W, float s, int ta);
};
static_assert(sizeof(DrawLean) == kTailSlotBytes, "five 16-byte words");

// Draws a warp computes ahead at once: two per lane (kTailSlots), or one where
// shared memory has no room for them (plan_tail).  A round's fixed cost (votes,
// the counters' shuffles, the timer) is shared by that many events.

// What the loops take of the run's parameters, by value.
struct LoneArgs {
  uint32_t max_events;
  int n_scat_max;
  int n_bins, imp;
  const uint64_t* spec_thr;
  const uint4* relax_tab;
  const float4* binf;
  uint32_t k0, k1;
};

__device__ __forceinline__ void load_bin_lone(Particle<float>& p, const float4* binf) {
  const float4 b = binf[p.bin];
  p.v = b.x;
  p.inv_v = b.y;
  p.lam = b.z;
}
// the two-phonon clock restarted (draw_d2)
__device__ __forceinline__ float d2_lone(const LoneArgs& A, int bin, float E2) {
  if (!A.imp) return Num<float>::inf();
  const float lam2 = A.binf[bin].w;
  return isinf(lam2) ? Num<float>::inf() : lam2 * E2;
}

// Reciprocal by the hardware's approximation.  a * rcp_hw(b) had the bits of
// __fdividef(a, b) in 2^33 random pairs with exponents -60 to 57, so a quotient
// can be split where b is known before a.  (The divisors here lie in that
// range: direction components, free paths and the pore's root in nm.  Beyond
// 2^126 __fdividef gives 0.)
__device__ __forceinline__ float rcp_hw(float b) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b));
  return r;
}
__device__ __forceinline__ float rcp_dir(float u) { return u == 0.0f ? 0.0f : rcp_hw(u); }

// contrib in fixed point (the value __float2ll_rn(contrib * kFx) has): the
// 32-bit conversion where it fits, off the FP64 pipe, whose latency (73 cycles
// against 18) a lone particle would wait out.
__device__ __forceinline__ long long fx_lone(float contrib) {
  const float s = contrib * kFx;
  return fabsf(s) < 2.0e9f ? (long long)__float2int_rn(s) : __float2ll_rn(s);
}

__device__ __forceinline__ void DrawLean::to_film(float LW, int W, float s, int ta) {
  const float seg = lam[0] != 0.0f ? fmaxf(LW * rlam[0], 0.0f) : Num<float>::big();
  float u[3];
  put3_cyclic<float>(u, W, lam[0], lam[1], lam[2]);
  const unsigned long long q = (unsigned long long)fx_lone((s * seg) * sel3(u, ta));
  rlam[2] = d_new;
  rlam[0] = __uint_as_float((uint32_t)q);
  rlam[1] = __uint_as_float((uint32_t)(q >> 32));
  riso[0] = lam[1];
  riso[1] = lam[2];
  riso[2] = lam[0];
  d_new = seg;
}

__device__ __forceinline__ void draw_lean(DrawLean& d, const GeoRun& g, const float4* binf, bool ext) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    d.riso[a] = rcp_dir(d.iso[a]);
    d.rlam[a] = rcp_dir(d.lam[a]);
  }
  d.d_new = binf[d.bin].z * d.E;
  uint32_t s = 0u;
#pragma unroll
  for (int f = 0; f < 6; ++f) s |= ((uint64_t)d.wx < g.pthr[f] ? 1u : 0u) << f;
  s |= ((uint64_t)d.wx < g.pthr_pore ? 1u : 0u) << 6;
  if (ext)
    for (int k = 0; k < g.n_inner; ++k) s |= ((uint64_t)d.wx < g.sthr[k] ? 1u : 0u) << (7 + k);
  d.spec = s;
}

// Internal wall k in shared memory: {nx, ny, x1, y1} and {tx, ty, |t|^2, -},
// t along the wall.
struct __align__(16) WallLean {
  float nx, ny, x1, y1, tx, ty, tt, pad;
  __device__ __forceinline__ void set(const GeoRun& g, int k) {
    if (k >= g.n_inner) {   // no wall: never met
      nx = ny = x1 = y1 = tx = ty = tt = pad = 0.0f;
      return;
    }
    nx = g.snxf[k];
    ny = g.snyf[k];
    x1 = g.sx1f[k];
    y1 = g.sy1f[k];
    tx = g.sx2f[k] - x1;
    ty = g.sy2f[k] - y1;
    tt = __fmaf_rn(tx, tx, __fmul_rn(ty, ty));
    pad = 0.0f;
  }
};

// What a flight's hit takes from its direction, per axis: the reciprocal, the
// face ahead (its coordinate, where the particle stands after meeting it, and
// its key: face ID, then type, axis and side), and the least distance (0, or
// "none" on an axis the direction does not move along).  The least key among
// the axes that reach the distance is the face the scan by ID finds.
struct LeanBox {
  float L[3], land_lo[3], land_hi[3];
  int key_lo[3], key_hi[3];

  static __device__ __forceinline__ int key_type(int k) { return (k >> 4) & 3; }
  static __device__ __forceinline__ int key_axis(int k) { return (k >> 1) & 3; }
  static __device__ __forceinline__ int key_face(int k) { return k >> 6; }

  __device__ __forceinline__ void load(const GeoRun& g) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      L[a] = g.Lf[a];
      const int f0 = axis_min_face(a), f1 = axis_max_face(a);
      const int t0 = g.type[f0], t1 = g.type[f1];
      land_lo[a] = t0 == MCBTE_FACE_PERIODIC ? L[a] : 0.0f;
      land_hi[a] = t1 == MCBTE_FACE_PERIODIC ? 0.0f : L[a];
      key_lo[a] = (f0 << 6) | (t0 << 4) | (a << 1);
      key_hi[a] = (f1 << 6) | (t1 << 4) | (a << 1) | 1;
    }
  }
};
struct LeanDir {
  float r[3], to[3], land[3], lo[3];
  int key[3];
  __device__ __forceinline__ void aim(const LeanBox& b, const float u[3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const bool up = u[a] > 0.0f;
      to[a] = up ? b.L[a] : 0.0f;
      land[a] = up ? b.land_hi[a] : b.land_lo[a];
      key[a] = up ? b.key_hi[a] : b.key_lo[a];
      lo[a] = u[a] == 0.0f ? Num<float>::big() : 0.0f;
    }
  }
};

// The tail kernel's events of one live particle: slot0 holds the draws of
// event p.e + 1, the slots end with event e_last.  Boxes with or without a
// pore, and with the extended physics internal walls, per-bin specularity and
// the two-phonon clock; gradients too.  (Detector regions, the N_scat_max
// curve and batches of geometries with walls take trace_slots.)  Returns at
// the particle's end, or ALIVE once the slots are used up.
// `walls`: the geometry's internal walls, to a multiple of four.
template <class Grad, class Tally, bool EXT, bool CELLS, bool PORE>
__device__ __forceinline__ int trace_lean(Particle<float>& p, const GeoRun& g, const WallLean* walls, const LoneArgs& A,
                                          const Tally& T, Grad& gr, const DrawLean* slot0, uint32_t e_last) {
  __builtin_assume(__isShared(slot0));   // shared-memory loads, not generic ones (half the latency)
  __builtin_assume(__isShared(walls));
  const uint32_t e0 = p.e;
  const uint32_t e_lim = e_last < A.max_events - 1u ? e_last : A.max_events - 1u;
  LeanBox box;
  box.load(g);
  const float cx = g.cxf, cy = g.cyf, r2 = g.r2f;
  LeanDir D;
#pragma unroll
  for (int a = 0; a < 3; ++a) D.r[a] = rcp_dir(p.u[a]);
  D.aim(box, p.u);
  float a2 = __fmaf_rn(p.u[0], p.u[0], __fmul_rn(p.u[1], p.u[1]));   // of the pore's quadratic
  float rlam = 0.0f;
  if (Grad::on) rlam = rcp_hw(p.lam);
  const int n_inner = EXT ? g.n_inner : 0;
  const unsigned perbin = EXT ? ((unsigned)g.fbin | ((unsigned)g.sbin << 7)) : 0u;
  uint64_t bin_thr = 0;
  if (EXT && perbin) bin_thr = A.spec_thr[p.bin];

  while (p.e < e_lim) {
    const DrawLean& d = slot0[p.e - e0];
    // nearest box face
    float c[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) c[a] = fmaxf((D.to[a] - p.x[a]) * D.r[a], D.lo[a]);
    const float bx = fminf(fminf(c[0], c[1]), c[2]);
    float db = bx;
    int surf = 0;   // 0 a box face, 6 the pore, 7 + k wall k
    if constexpr (PORE) {
      const float dx = p.x[0] - cx, dy = p.x[1] - cy;
      const float b = __fmaf_rn(dx, p.u[0], __fmul_rn(dy, p.u[1]));
      const float cc = __fmaf_rn(dx, dx, __fmul_rn(dy, dy)) - r2;
      const float disc = __fmaf_rn(b, b, -__fmul_rn(a2, cc));
      const bool hit = a2 > 0.0f && b < 0.0f && disc >= 0.0f;
      const float dp = fmaxf(cc * rcp_hw(sqrt_approx(fmaxf(disc, 0.0f)) - b), 0.0f);
      const bool take = hit && dp < db;
      db = take ? dp : db;
      surf = take ? 6 : surf;
    }
    if constexpr (EXT) {
      for (int k0 = 0; k0 < n_inner; k0 += 4) {
        // four walls at a time, their constants read together
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const WallLean w = walls[k0 + j];
          const float un = __fmaf_rn(p.u[0], w.nx, __fmul_rn(p.u[1], w.ny));
          const float ax = p.x[0] - w.x1, ay = p.x[1] - w.y1;
          const float dn = __fmaf_rn(ax, w.nx, __fmul_rn(ay, w.ny));
          const float dw = fmaxf(dn * rcp_hw(-un), 0.0f);
          const float hs = __fmaf_rn(__fmaf_rn(dw, p.u[0], p.x[0]) - w.x1, w.tx,
                                     __fmul_rn(__fmaf_rn(dw, p.u[1], p.x[1]) - w.y1, w.ty));
          const bool take = un < 0.0f && !(dn < -1e-4f) && !(hs < 0.0f || hs > w.tt) && dw < db;
          db = take ? dw : db;
          surf = take ? 7 + k0 + j : surf;
        }
      }
    }
    const bool relax = EXT ? (p.d_rel < db && p.d_rel <= p.d2) : p.d_rel < db;
    const bool relax2 = EXT && !relax && p.d2 < db;
    const float seg = relax ? p.d_rel : (relax2 ? p.d2 : db);
    float contrib;
    if constexpr (CELLS) {
      contrib = T.segment(p, seg);
    } else {
      contrib = (p.s * seg) * sel3(p.u, T.ta);
      p.Xq += fx_lone(contrib);
    }
    if (Grad::on) gr.flight(relax, (double)(seg * rlam), 0.0, contrib);
#pragma unroll
    for (int a = 0; a < 3; ++a) p.x[a] = __fmaf_rn(seg, p.u[a], p.x[a]);
    ++p.e;
    if (__builtin_expect(relax || relax2, 0)) {
      if (relax2) {
        p.d_rel = p.d_rel - seg;
      } else {
        ++p.n_relax;
        if (A.n_scat_max > 0 && p.n_relax >= A.n_scat_max) return STEP_DONE;
        T.period_end(p);
        p.bin = d.bin;
        p.d_rel = d.d_new;
        load_bin_lone(p, A.binf);
        if (EXT && perbin) bin_thr = A.spec_thr[p.bin];
        if (Grad::on) {
          rlam = rcp_hw(p.lam);
          gr.resampled(p.bin, T.X(p));
        }
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        p.u[a] = d.iso[a];
        D.r[a] = d.riso[a];
      }
      if constexpr (EXT) p.d2 = d2_lone(A, p.bin, d.E2);
    } else {
      p.d_rel = p.d_rel - seg;
      if constexpr (EXT) p.d2 = p.d2 - seg;
      if (surf == 0) {
        const int k = min(min(c[0] == bx ? D.key[0] : 0x7fffffff, c[1] == bx ? D.key[1] : 0x7fffffff),
                          c[2] == bx ? D.key[2] : 0x7fffffff);
        const int a = LeanBox::key_axis(k);
#pragma unroll
        for (int b = 0; b < 3; ++b) p.x[b] = b == a ? D.land[b] : p.x[b];
        const int ty = LeanBox::key_type(k);
        if (ty == MCBTE_FACE_PERIODIC) continue;
        if (ty == MCBTE_FACE_ISOTHERMAL) return STEP_ABSORBED;
        const int f = LeanBox::key_face(k);
        const bool mx = (k & 1) != 0;
        const bool spec = (EXT && ((perbin >> f) & 1u)) ? (uint64_t)d.wx < bin_thr : ((d.spec >> f) & 1u) != 0u;
        float ud[3], rd[3];
        put3_cyclic<float>(ud, a, mx ? -d.lam[0] : d.lam[0], d.lam[1], d.lam[2]);
        put3_cyclic<float>(rd, a, mx ? -d.rlam[0] : d.rlam[0], d.rlam[1], d.rlam[2]);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          p.u[b] = spec ? (b == a ? -p.u[b] : p.u[b]) : ud[b];
          D.r[b] = spec ? (b == a ? -D.r[b] : D.r[b]) : rd[b];
        }
      } else {
        float nx, ny;
        bool spec;
        if (EXT && (!PORE || surf >= 7)) {
          const WallLean w = walls[surf - 7];
          nx = w.nx;
          ny = w.ny;
          const float dn = __fmaf_rn(p.x[0] - w.x1, nx, __fmul_rn(p.x[1] - w.y1, ny));
          p.x[0] = __fmaf_rn(-dn, nx, p.x[0]);
          p.x[1] = __fmaf_rn(-dn, ny, p.x[1]);
          spec = ((perbin >> surf) & 1u) ? (uint64_t)d.wx < bin_thr : ((d.spec >> surf) & 1u) != 0u;
        } else {
          nx = p.x[0] - cx;
          ny = p.x[1] - cy;
          const float il = rsqrtf(__fmaf_rn(nx, nx, __fmul_rn(ny, ny)));
          nx = nx * il;
          ny = ny * il;
          spec = ((d.spec >> 6) & 1u) != 0u;
          if (Grad::on) {
            spec = gr.pore_branch(spec, g.p_pore, 0.0,
                                  [&] { return DrawSlot{&d}.mv(make_uint4(0u, 0u, 0u, 0u), 0u, 0u); });
            gr.pore_hit(p);
          }
        }
        const float two_un = 2.0f * __fmaf_rn(p.u[0], nx, __fmul_rn(p.u[1], ny));
        const float s0 = __fmaf_rn(-two_un, nx, p.u[0]);
        const float s1 = __fmaf_rn(-two_un, ny, p.u[1]);
        const float l0 = __fmaf_rn(d.lam[0], nx, -__fmul_rn(d.lam[1], ny));
        const float l1 = __fmaf_rn(d.lam[0], ny, __fmul_rn(d.lam[1], nx));
        p.u[0] = spec ? s0 : l0;
        p.u[1] = spec ? s1 : l1;
        p.u[2] = spec ? p.u[2] : d.lam[2];
        D.r[0] = rcp_dir(p.u[0]);
        D.r[1] = rcp_dir(p.u[1]);
        D.r[2] = spec ? D.r[2] : d.rlam[2];
      }
    }
    D.aim(box, p.u);
    a2 = __fmaf_rn(p.u[0], p.u[0], __fmul_rn(p.u[1], p.u[1]));
  }
  return p.e + 1u >= A.max_events ? STEP_TRUNCATED : STEP_ALIVE;
}

// Events per flight of a film's particle: a diffuse flight across it meets
// LW / LA + LW / LB periodic faces in the mean, each of them an event number
// (and a draw computed ahead that nothing reads).  0: not a film.
__device__ __forceinline__ float film_events(const GeoRun& g, unsigned um) {
  const int W = um == 3u ? 2 : (um == 5u ? 1 : (um == 6u ? 0 : -1));
  if (W < 0) return 0.0f;
  const float LW = geo_L<float>(g, W), LA = geo_L<float>(g, (W + 1) % 3), LB = geo_L<float>(g, (W + 2) % 3);
  return 1.0f + LW * rcp_hw(LA) + LW * rcp_hw(LB);
}
// A round of draws ahead costs a warp about as much as four flights that draw
// inline, so thick films, whose slots end before that, take no slots (silicon,
// 1e5 particles, us with the line at 1, 2, 4, 8 and 16 flights: film of 300 nm
// 613, 617, 612, 622, 726; 600 nm 530, 520, 519, 490, 485; 1000 nm 434, 434,
// 369, 365, 366; 20 films of 10 to 10 000 nm 4284, 4284, 4284, 4733, 4728).  The
// warp decides for all it holds, by most of its live particles.
constexpr float kInlineFlights = 4.0f;
// Flights of a round without slots, then the warp votes again (film of 600 nm
// with 8, 32 and 128: 542, 519, 512 us; of 150 nm 888, 894, 924).
constexpr float kInlineRound = 32.0f;

// The tail loop of a film: a box without pore or walls whose flights run
// through the two periodic axes (forward run without cell tallies or extended
// physics), so that the faces left are the pair across axis W.  A flight from
// wall to wall has the length and the tally its wall's draws give it, wherever
// it starts along the film: both are in the draws (seg, cq), and the chain
// from flight to flight holds two additions along the film, the relaxation
// clock and the fold at the periodic faces.  The crossings advance the event
// number, so the event that ends a flight may lie past the slots and then
// takes its draws inline (the same bits).  nslots: the draws at slot0, or 0 to
// take every event's inline up to event e_last.
template <int W, class Tally>
__device__ __forceinline__ int trace_film(Particle<float>& p, const GeoRun& g, const LoneArgs& R, const Tally& T,
                                          const DrawLean* slot0, uint32_t nslots, uint32_t e_last) {
  constexpr int A = (W + 1) % 3, B = (W + 2) % 3;   // along the film; put3_cyclic's order
  const uint32_t e0 = p.e;
  const float LA = g.Lf[A], LB = g.Lf[B], LW = g.Lf[W];
  const int f_lo = axis_min_face(W), f_hi = axis_max_face(W);
  const bool iso_lo = g.type[f_lo] == MCBTE_FACE_ISOTHERMAL, iso_hi = g.type[f_hi] == MCBTE_FACE_ISOTHERMAL;
  const bool across = T.ta == W;   // the tally axis: its component changes sign with the wall
  const float s = p.s;
  // the flight ahead: its length to the wall and its tally
  float db;
  bool up;
  long long cq;
  __builtin_assume(__isShared(slot0));
  auto aim = [&]() {
    up = p.u[W] > 0.0f;
    db = p.u[W] != 0.0f ? fmaxf(((up ? LW : 0.0f) - p.x[W]) * rcp_hw(p.u[W]), 0.0f) : Num<float>::big();
    cq = fx_lone((s * db) * sel3(p.u, T.ta));
  };
  aim();
  // the flight ahead runs from wall to wall (its length and tally then stay
  // under a specular reflection, in every bit)
  bool full = p.x[W] == (up ? 0.0f : LW);
  // Flights from wall to wall that do not relax, in a loop of their own with
  // the next draws read ahead.  An unsigned comparison of the bits takes
  // 0 <= x < L in one test; a flight past one periodic face is folded here
  // (x -+ L, the value fold_periodic gives clear of its quotient's roundings),
  // a specular reflection keeps the flight's length and tally.
  const uint32_t iLA = __float_as_uint(LA), iLB = __float_as_uint(LB);
  const bool quick = nslots != 0u && !across && !iso_lo && !iso_hi;
  const uint32_t e_lim = e_last < R.max_events - 1u ? e_last : R.max_events - 1u;
  for (;;) {
    if (quick && db < Num<float>::big()) {
      uint32_t hi = up ? 1u << f_hi : 1u << f_lo;
      const uint32_t both = (1u << f_hi) ^ (1u << f_lo);
      uint32_t e = p.e;
      float x = p.x[A], y = p.x[B], ua = p.u[A], ub = p.u[B], l0 = fabsf(p.u[W]), dr = p.d_rel;
      long long X = p.Xq;
      bool moved = false;
      while (e < e_lim) {
        const DrawLean* d = slot0 + (e - e0);
        float4 nx = d->film_flight();
        long long nq = d->film_tally();
        uint32_t sp = d->spec;
        float xn = __fmaf_rn(db, ua, x), yn = __fmaf_rn(db, ub, y);
        if (dr < db) break;
        uint32_t n = 0u;
        if (!(__float_as_uint(xn) < iLA && __float_as_uint(yn) < iLB)) {
          bool fold = true;
          if (!(__float_as_uint(xn) < iLA)) {
            const float r = xn + (xn < 0.0f ? LA : -LA);
            fold = xn > -0.999f * LA && xn < 1.999f * LA && __float_as_uint(r) < iLA;
            xn = r;
            n = 1u;
          }
          if (!(__float_as_uint(yn) < iLB)) {
            const float r = yn + (yn < 0.0f ? LB : -LB);
            fold = fold && yn > -0.999f * LB && yn < 1.999f * LB && __float_as_uint(r) < iLB;
            yn = r;
            ++n;
          }
          if (!fold) {
            // past more than one period (films thicker than their period)
            float q[3];
            q[W] = 0.0f;
            q[A] = __fmaf_rn(db, ua, x);
            q[B] = __fmaf_rn(db, ub, y);
            n = fold_periodic(q, g.Lf, (1u << A) | (1u << B));
            xn = q[A];
            yn = q[B];
          }
          if (n >= e_lim - e) break;
          d += n;
          nx = d->film_flight();
          nq = d->film_tally();
          sp = d->spec;
        }
        const bool spec = (sp & hi) != 0u;
        if (spec && !full) break;
        X += cq;
        dr = dr - db;
        x = xn;
        y = yn;
        ua = spec ? ua : nx.x;
        ub = spec ? ub : nx.y;
        l0 = spec ? l0 : nx.z;
        db = spec ? db : nx.w;
        cq = spec ? cq : nq;
        hi ^= both;
        full = moved = true;
        e += n + 1u;
      }
      if (moved) {
        up = hi == 1u << f_hi;
        p.e = e;
        p.Xq = X;
        p.d_rel = dr;
        p.x[A] = x;
        p.x[B] = y;
        p.x[W] = up ? 0.0f : LW;
        p.u[A] = ua;
        p.u[B] = ub;
        p.u[W] = up ? l0 : -l0;
        if (e >= e_last) return STEP_ALIVE;
      }
    }
    if (p.e + 1u >= R.max_events) return STEP_TRUNCATED;
    const bool relax = p.d_rel < db;
    const float seg = relax ? p.d_rel : db;
    uint32_t n = 0u;
    p.x[A] = __fmaf_rn(seg, p.u[A], p.x[A]);
    p.x[B] = __fmaf_rn(seg, p.u[B], p.x[B]);
    if (!(p.x[A] >= 0.0f && p.x[A] < LA && p.x[B] >= 0.0f && p.x[B] < LB)) {
      n = fold_periodic(p.x, g.Lf, (1u << A) | (1u << B));
      if (n >= R.max_events - 1u - p.e) {
        p.Xq += relax ? fx_lone((s * seg) * sel3(p.u, T.ta)) : cq;
        p.e = R.max_events - 1u;
        return STEP_TRUNCATED;
      }
    }
    const uint32_t si = p.e + n - e0;
    const DrawLean* d = slot0 + (si < nslots ? si : 0u);
    p.e += n + 1u;
    if (relax) {
      p.Xq += fx_lone((s * seg) * sel3(p.u, T.ta));
      p.x[W] = __fmaf_rn(seg, p.u[W], p.x[W]);
      ++p.n_relax;
      if (R.n_scat_max > 0 && p.n_relax >= R.n_scat_max) return STEP_DONE;
      T.period_end(p);
      if (si < nslots) {
        p.bin = d->bin;
        p.d_rel = d->film_d_new();
#pragma unroll
        for (int a = 0; a < 3; ++a) p.u[a] = d->iso[a];
        load_bin_lone(p, R.binf);
      } else {
        Draw32 f;
        draw_words(f, philox(make_uint4(p.pid, (uint32_t)p.g, p.e, 0u), R.k0, R.k1), R.relax_tab, R.n_bins);
        p.bin = f.bin;
#pragma unroll
        for (int a = 0; a < 3; ++a) p.u[a] = f.iso[a];
        load_bin_lone(p, R.binf);
        p.d_rel = p.lam * f.E;
      }
      aim();
      full = false;
    } else {
      p.Xq += cq;
      p.d_rel = p.d_rel - seg;
      p.x[W] = up ? LW : 0.0f;
      full = true;
      if (up ? iso_hi : iso_lo) return STEP_ABSORBED;
      if (si < nslots) {
        const bool spec = ((d->spec >> (up ? f_hi : f_lo)) & 1u) != 0u;
        if (spec) {
          p.u[W] = -p.u[W];
          aim();
        } else {
          p.u[W] = up ? -d->lam[0] : d->lam[0];
          p.u[A] = d->lam[1];
          p.u[B] = d->lam[2];
          db = d->d_new;
          cq = up && across ? -d->film_tally() : d->film_tally();
          up = !up;   // (lam[0] >= 2^-12)
        }
      } else {
        Draw32 f;
        draw_words(f, philox(make_uint4(p.pid, (uint32_t)p.g, p.e, 0u), R.k0, R.k1), R.relax_tab, R.n_bins);
        if ((uint64_t)f.wx < g.pthr[up ? f_hi : f_lo]) {
          p.u[W] = -p.u[W];
        } else {
          p.u[W] = up ? -f.lam[0] : f.lam[0];
          p.u[A] = f.lam[1];
          p.u[B] = f.lam[2];
        }
        aim();
      }
    }
    if (p.e >= e_last) return STEP_ALIVE;
  }
}

// A round of a particle's events by one of the loops.  Each is out of line, on
// copies of the particle, the tally and the estimator: inlined into the tail
// kernel the same loops ran longer (pore lattice 571 cycles an event, 451 out
// of line and 344 alone in a small kernel), their instructions spread over a
// kernel that a lone warp then fetches line by line.
// LOOP: 0-2 a film across that axis, 3 a box, 4 a box with a pore.
template <int LOOP, class Grad, class Tally, bool EXT, bool CELLS>
static __device__ __noinline__ int trace_round(Particle<float>* pp, const GeoRun* g, const WallLean* walls, LoneArgs A,
                                               const Tally* tt, Grad* gg, const DrawLean* slot0, uint32_t nslots,
                                               uint32_t e_last) {
  Particle<float> p = *pp;
  const Tally T = *tt;
  Grad gr = *gg;
  int out;
  if constexpr (LOOP < 3) out = trace_film<LOOP>(p, *g, A, T, slot0, nslots, e_last);
  else out = trace_lean<Grad, Tally, EXT, CELLS, LOOP == 4>(p, *g, walls, A, T, gr, slot0, e_last);
  *pp = p;
  if (Grad::on) *gg = gr;
  return out;
}

// The loop of the particle's geometry; `um`: the unfolded periodic axes where
// they are a film's two, else 0.
template <class Grad, class Tally, bool EXT, bool CELLS>
__device__ __forceinline__ int trace_alone(Particle<float>& p, const GeoRun& g, const WallLean* walls, const LoneArgs& A,
                                           const Tally& T, Grad& gr, const DrawLean* slot0, uint32_t nslots,
                                           uint32_t e_last, unsigned um) {
  Particle<float> q = p;
  const Tally Tq = T;
  Grad gq = gr;
  int out = STEP_ALIVE;
#define MCBTE_LOOP(k) out = trace_round<k, Grad, Tally, EXT, CELLS>(&q, &g, walls, A, &Tq, &gq, slot0, nslots, e_last)
  bool film = false;
  if constexpr (!CELLS && !EXT && !Grad::on) {
    film = um != 0u;
    if (um == 3u) MCBTE_LOOP(2);
    else if (um == 5u) MCBTE_LOOP(1);
    else if (um == 6u) MCBTE_LOOP(0);
  }
  if (!film) {
    if (g.pore) MCBTE_LOOP(4);
    else MCBTE_LOOP(3);
  }
#undef MCBTE_LOOP
  p = q;
  if (Grad::on) gr = gq;
  return out;
}

}  // namespace mcbte
