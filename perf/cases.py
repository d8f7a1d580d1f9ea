"""Performance cases of the deviational phonon Monte Carlo library.

Each case is one call (or one forward and backward) of the public entry
points, at the sizes the configurations, tests and benchmark of this
repository use.  ``listed()`` names the fixed ones, ``draw()`` gives more of
the same ranges, ``exact()`` traces wall-to-wall cases again in 64-bit torch.
"""
from __future__ import annotations

import math
from dataclasses import dataclass, replace
from typing import Optional, Sequence

import numpy as np
import torch

from paper_2104_03573_gb300 import _lib as L
from paper_2104_03573_gb300 import api, autograd, batch

ISOTHERMAL, ADIABATIC, PERIODIC = 0, 1, 2
NM = 1e-9


# ---------------------------------------------------------------- inputs
@dataclass
class Material:
    """Material columns in SI units, as the library takes them."""
    omega: np.ndarray
    v: np.ndarray
    tau: np.ndarray
    D: Optional[np.ndarray] = None
    domega: Optional[np.ndarray] = None
    C: Optional[np.ndarray] = None
    T_lin: float = 300.0
    tau_imp: Optional[np.ndarray] = None
    spec_bin: Optional[np.ndarray] = None

    def scaled_tau(self, log_scale):
        return replace(self, tau=self.tau * np.exp(np.asarray(log_scale, dtype=np.float64)))


@dataclass
class Box:
    """Geometry description, as the library takes it."""
    L: Sequence[float]
    face_type: Sequence[int]
    face_T: Sequence[float] = (0.0,) * 6
    face_p: Sequence[float] = (0.0,) * 6
    T_eq: float = 300.0
    grad_T: Sequence[float] = (0.0, 0.0, 0.0)
    pore: bool = False
    pore_c: Sequence[float] = (0.0, 0.0)
    pore_r: float = 0.0
    pore_p: float = 0.0
    gauss: bool = False
    gauss_c: Sequence[float] = (0.0, 0.0, 0.0)
    gauss_sigma: float = 0.0
    gauss_dT: float = 0.0
    inner: Sequence = ()
    inner_n: Sequence = ()
    inner_p: Sequence[float] = ()


def gray(mfp, v=6000.0, tau=None):
    return Material(omega=np.array([1e13]), v=np.array([v]), tau=np.array([tau or mfp / v]), C=np.array([1e6]))


def silicon(per_branch=1000, T=300.0):
    """Silicon-like dispersion (one LA, two TA branches), Holland-type tau."""
    kmax = 2.0 * math.pi / 5.43e-10
    cols = []
    for wmax in (7.7e13, 2.8e13, 2.8e13):
        dw = wmax / per_branch
        w = (np.arange(per_branch) + 0.5) * dw
        k = (2.0 * kmax / math.pi) * np.arcsin(w / wmax)
        v = wmax * (math.pi / (2.0 * kmax)) * np.cos(math.pi * k / (2.0 * kmax))
        tau = 1.0 / (1.32e-45 * w ** 4 + 1.73e-19 * w ** 2 * T * math.exp(-137.0 / T))
        cols.append((w, v, tau, k * k / (2.0 * math.pi ** 2 * v), np.full_like(w, dw)))
    w, v, tau, D, dw = (np.concatenate(c) for c in zip(*cols))
    return Material(omega=w, v=v, tau=tau, D=D, domega=dw, T_lin=T)


def slab(length, dT, lateral):
    """Isothermal walls at z = 0 and z = length, periodic x and y."""
    ft = [PERIODIC] * 4 + [ISOTHERMAL] * 2
    return Box(L=(lateral, lateral, length), face_type=ft, face_T=[0.0] * 4 + [300.0 + dT, 300.0 - dT])


def film(d, W=100 * NM, p=0.0):
    """Periodic x and y, adiabatic z walls, control gradient along y."""
    return Box(L=(W, W, d), face_type=[PERIODIC] * 4 + [ADIABATIC] * 2, face_p=[0.0] * 4 + [p, p],
               grad_T=(0.0, -1e6, 0.0))


def pore_film(W, porosity, thickness, p_pore=0.0):
    return replace(film(thickness, W), pore=True, pore_c=(0.5 * W, 0.5 * W),
                   pore_r=W * math.sqrt(porosity / math.pi), pore_p=p_pore)


def nanomesh(W, pore, thickness):
    """A square pore in a square cell: four internal walls that take the
    material's per-bin specularity, as the film's faces do."""
    a, b = 0.5 * (W - pore), 0.5 * (W + pore)
    return replace(film(thickness, W, p=-1.0), inner=[(a, a, b, a), (b, a, b, b), (b, b, a, b), (a, b, a, a)],
                   inner_n=[(0.0, -1.0), (1.0, 0.0), (0.0, 1.0), (-1.0, 0.0)], inner_p=[-1.0] * 4)


def hot_spot_box():
    return Box(L=(2e-6, 2e-6, 1e-6), face_type=[ADIABATIC] * 6, gauss=True, gauss_c=(1e-6, 1e-6, 1e-6),
               gauss_sigma=100 * NM, gauss_dT=1.0)


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: a quick look at a gray slab, launches and latency
        {"name": "gray_slab_4k", "kind": "slab", "gray": True, "n": 4096, "nm": 100.0, "cells": 50,
         "per_bin": False, "axis_flux": False, "fp64": False},
        # the gray validation slab at its usual size
        {"name": "gray_slab_100k", "kind": "slab", "gray": True, "n": 100_000, "nm": 100.0, "cells": 50,
         "per_bin": False, "axis_flux": False, "fp64": False},
        # the headline: silicon-like cross-plane film, spectral flux, axial cell flux
        {"name": "si_slab_10m", "kind": "slab", "gray": False, "n": 10_000_000, "nm": 1000.0, "cells": 50,
         "per_bin": True, "axis_flux": True, "fp64": False},
        # the reference precision, checked particle by particle against a CPU code
        {"name": "gray_slab_fp64_100k", "kind": "slab", "gray": True, "n": 100_000, "nm": 100.0, "cells": 50,
         "per_bin": False, "axis_flux": False, "fp64": True},
        # the reference precision over the full spectrum, an odd particle count
        {"name": "si_slab_fp64_301k", "kind": "slab", "gray": False, "n": 301_307, "nm": 1000.0, "cells": 50,
         "per_bin": True, "axis_flux": False, "fp64": True},
        # conductivity against thickness: a batch of films replayed as a graph
        {"name": "films_64", "kind": "films", "films": 64, "scale": 0.1, "thin_nm": 10.0, "thick_nm": 10000.0},
        # conductivity of a nanoporous film
        {"name": "pore_film_5m", "kind": "pore", "n": 5_000_000, "W_nm": 100.0, "porosity": 0.25, "nm": 200.0,
         "p": 0.0, "grad": False, "dirs": 0, "fp64": False},
        # its sensitivities to every bin's relaxation time and to the pore walls
        {"name": "pore_grad_2m", "kind": "pore", "n": 2_000_000, "W_nm": 100.0, "porosity": 0.25, "nm": 200.0,
         "p": 0.0, "grad": True, "dirs": 0, "fp64": False},
        # one step of a calibration loop through torch.autograd, new tau each step
        {"name": "kappa_step_100k", "kind": "kappa", "n": 100_000, "W_nm": 100.0, "porosity": 0.25, "nm": 200.0,
         "p": 0.3},
        # extended physics: square pores, frequency-dependent specular walls
        {"name": "nanomesh_301k", "kind": "mesh", "n": 301_307, "W_nm": 34.0, "pore_nm": 11.0, "nm": 22.0},
        # laser-pulse relaxation: a hot spot on the 3-D grid, 200 snapshots
        {"name": "hot_spot_10m", "kind": "spot", "n": 10_000_000, "nx": 64, "ny": 64, "nz": 32, "times": 200,
         "average": False, "fp64": False},
        # a ballistic transient between two walls, few snapshots
        {"name": "wall_pulse_200k", "kind": "walls", "n": 200_000, "cells": 30, "times": 6},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["gray", "gray", "si", "si", "films", "pore", "pore", "kappa", "mesh", "spot", "walls"])
    if kind == "gray":
        fp64 = rng.random() < 0.4
        return {"kind": "slab", "gray": True, "n": int(_log(rng, 1000, 200_000 if fp64 else 2_000_000)),
                "nm": round(_log(rng, 20.0, 400.0), 2), "cells": rng.choice([0, 7, 50, 101]),
                "per_bin": rng.random() < 0.3, "axis_flux": rng.random() < 0.5, "fp64": fp64}
    if kind == "si":
        fp64 = rng.random() < 0.4
        return {"kind": "slab", "gray": False, "n": int(_log(rng, 2000, 100_000 if fp64 else 5_000_000)),
                "nm": round(_log(rng, 100.0, 1500.0), 2), "cells": rng.choice([0, 7, 50, 101]),
                "per_bin": rng.random() < 0.7, "axis_flux": rng.random() < 0.5, "fp64": fp64}
    if kind == "films":
        return {"kind": "films", "films": rng.randint(1, 64), "scale": round(_log(rng, 0.003, 0.06), 5),
                "thin_nm": round(_log(rng, 20.0, 200.0), 2), "thick_nm": round(_log(rng, 500.0, 10000.0), 2)}
    if kind == "pore":
        grad = rng.random() < 0.5
        fp64 = rng.random() < 0.2
        return {"kind": "pore", "n": int(_log(rng, 2000, 20_000 if fp64 else 1_000_000)),
                "W_nm": round(_log(rng, 50.0, 300.0), 2), "porosity": round(rng.uniform(0.05, 0.4), 3),
                "nm": round(_log(rng, 50.0, 500.0), 2), "p": rng.choice([0.0, 0.0, round(rng.uniform(0.1, 0.9), 3)]),
                "grad": grad, "dirs": rng.choice([0, 3]) if grad else 0, "fp64": fp64}
    if kind == "kappa":
        return {"kind": "kappa", "n": int(_log(rng, 2000, 400_000)), "W_nm": round(_log(rng, 50.0, 300.0), 2),
                "porosity": round(rng.uniform(0.05, 0.4), 3), "nm": round(_log(rng, 50.0, 500.0), 2),
                "p": round(rng.uniform(0.1, 0.9), 3)}
    if kind == "mesh":
        W = round(_log(rng, 30.0, 100.0), 2)
        return {"kind": "mesh", "n": int(_log(rng, 2000, 300_000)), "W_nm": W,
                "pore_nm": round(W * rng.uniform(0.2, 0.5), 2), "nm": round(_log(rng, 22.0, 100.0), 2)}
    if kind == "spot":
        fp64 = rng.random() < 0.2
        return {"kind": "spot", "n": int(_log(rng, 5000, 50_000 if fp64 else 3_000_000)), "nx": rng.randint(5, 64),
                "ny": rng.randint(5, 64), "nz": rng.randint(3, 32), "times": rng.randint(3, 200),
                "average": rng.random() < 0.3, "fp64": fp64}
    return {"kind": "walls", "n": int(_log(rng, 2000, 2_000_000)), "cells": rng.randint(5, 100),
            "times": rng.randint(2, 40)}


def _film_batch(case):
    """Thicknesses and particle counts of the batch: the counts spread over
    two decades, as an adaptive sweep asks for them."""
    k = case["films"]
    u = np.random.default_rng(1004).uniform(0.0, 1.0, size=k)
    n = [max(1, int(round(case["scale"] * 1e5 * 100.0 ** x))) for x in u]
    ratio = case["thick_nm"] / case["thin_nm"]
    d = [case["thin_nm"] * NM * ratio ** (f / max(1, k - 1)) for f in range(k)]
    return d, n


def _wall_times(case):
    return 900e-12 * (np.arange(1, case["times"] + 1) / case["times"]) ** 2


def _slab_parts(case):
    mat = gray(100 * NM) if case["gray"] else silicon()
    return mat, slab(case["nm"] * NM, 0.5, 100 * NM if case["gray"] else 1e-6)


def _wall_parts():
    return gray(None, v=12360.0, tau=1.0), slab(3e-6, 3.0, 3e-6)


def prepare(case, seed):
    kind = case["kind"]
    key = 1 + seed * 2654435761 % (1 << 40)
    precision = L.FP64_PLAIN if case.get("fp64") else L.FP32_TRACE
    if kind == "slab":
        mat, geo = _slab_parts(case)
        cfg = api.SteadyConfig(seed=key, precision=precision, n_cells=case["cells"], per_bin=case["per_bin"],
                               cell_flux_axis=case["axis_flux"])
        return {"case": case, "mat": api.Material(mat), "geo": api.Geometry(geo), "cfg": cfg}
    if kind == "films":
        d, n = _film_batch(case)
        cfg = api.SteadyConfig(seed=key, tally_axis=1, per_bin=True, n_scat_max=10)
        m = api.Material(silicon())
        return {"case": case, "key": key,
                "graph": batch.GraphBatch(m, [api.Geometry(film(x)) for x in d], n, cfg, tune=False)}
    if kind == "pore":
        geo = pore_film(case["W_nm"] * NM, case["porosity"], case["nm"] * NM, case["p"])
        cfg = api.SteadyConfig(seed=key, precision=precision, tally_axis=1, per_bin=True, n_scat_max=10)
        m = api.Material(silicon())
        dirs = None
        if case["dirs"]:
            gen = np.random.default_rng(seed)
            dirs = torch.from_numpy(gen.normal(size=(case["dirs"], m.n_bins)) / math.sqrt(m.n_bins))
        return {"case": case, "mat": m, "geo": api.Geometry(geo), "cfg": cfg, "dirs": dirs}
    if kind == "kappa":
        mat = silicon()
        geo = pore_film(case["W_nm"] * NM, case["porosity"], case["nm"] * NM, case["p"])
        gen = np.random.default_rng(seed)
        s = torch.from_numpy(0.05 * gen.normal(size=mat.omega.size)).requires_grad_()
        p = torch.tensor(case["p"], dtype=torch.float64, requires_grad=True)
        cfg = api.SteadyConfig(seed=key, tally_axis=1, n_scat_max=10)
        return {"case": case, "s": s, "p": p, "mat": mat, "geo": geo, "cfg": cfg}
    if kind == "mesh":
        mat = silicon()
        mat = replace(mat, spec_bin=(mat.omega <= 2e12 * 2.0 * math.pi).astype(np.float64))
        geo = nanomesh(case["W_nm"] * NM, case["pore_nm"] * NM, case["nm"] * NM)
        cfg = api.SteadyConfig(seed=key, tally_axis=1, per_bin=True, n_scat_max=10)
        return {"case": case, "mat": api.Material(mat), "geo": api.Geometry(geo), "cfg": cfg}
    if kind == "spot":
        t = 2e-9 / case["times"] * np.arange(1, case["times"] + 1)
        grid = (case["nx"], case["ny"], case["nz"])
        mat, geo, average = silicon(), hot_spot_box(), case["average"]
    else:
        t, grid, average = _wall_times(case), (1, 1, case["cells"]), False
        mat, geo = _wall_parts()
    cfg = api.TransientConfig(seed=key, t_max=float(t[-1]), t_meas=t, grid=grid, precision=precision,
                              time_average=average)
    return {"case": case, "mat": api.Material(mat), "geo": api.Geometry(geo), "cfg": cfg,
            "out": api.TransientOutputs(len(t), grid, case["n"])}


def _steady_result(out):
    return {"stats": out.stats, "T": out.T, "q": out.q, "q_bin": out.q_bin}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "films":
        return _steady_result(state["graph"].replay(state["key"]))
    if kind == "kappa":
        state["s"].grad = state["p"].grad = None
        k = autograd.kappa(state["s"], state["p"], state["mat"], state["geo"], case["n"], state["cfg"])
        k.backward()
        return {"kappa": k, "dtau": state["s"].grad, "dp": state["p"].grad}
    if kind in ("spot", "walls"):
        out = api.run_transient(state["mat"], state["geo"], case["n"], state["cfg"], out=state["out"])
        return {"tally": out.tally, "stats": out.stats}
    if kind == "pore" and case["grad"]:
        out, g = api.grad(state["mat"], state["geo"], case["n"], state["cfg"], dirs=state["dirs"])
        res = _steady_result(out)
        res.update(dtau=g.dkappa_dlogtau, dp=g.dkappa_dp)
        if case["dirs"]:
            res["ddir"] = g.dkappa_dir
        return res
    return _steady_result(api.run_steady(state["mat"], [state["geo"]], [case["n"]], state["cfg"]))


# ---------------------------------------------------------------- least work
def work(case):
    """Material tables and outputs once through memory; per event about 200
    operations (one Philox block, the logarithm, roots and sines of a new
    direction, the first hit and the tallies), per snapshot about 20."""
    kind, n = case["kind"], case.get("n", 0)
    bins = 1 if case.get("gray") or kind == "walls" else 3000
    out = 16 * 8
    # events per particle as such runs count them
    if kind == "slab":
        events = n * (2.0 + (0.04 if case["gray"] else 0.064) * case["nm"])
        out += 32 * case["cells"] + (8 * bins if case["per_bin"] else 0)
    elif kind == "films":
        d, per = _film_batch(case)
        events = 18.0 * sum(per)
        out = len(d) * (16 * 8 + 8 * bins)
    elif kind in ("pore", "kappa"):
        events = n * (10.0 + 1150.0 / case["W_nm"])
        out += 8 * bins * (2 if kind == "kappa" or case["grad"] else 1)
    elif kind == "mesh":
        events = n * 1440.0 / case["W_nm"]
        out += 8 * bins
    elif kind == "spot":
        events = n * 140.0 + 0.1 * n * case["times"]
        out += 32 * case["nx"] * case["ny"] * case["nz"] * case["times"]
    else:
        events = n * 2.7 + 0.1 * n * case["times"]
        out += 32 * case["cells"] * case["times"]
    return {"bytes": 16 * 5 * bins + out, "flops": 200.0 * events}


# ---------------------------------------------------------------- 64-bit values
def _alias(weights):
    """Walker table by Vose's lists: (thresholds * 2^-64 as integers, alias)."""
    total = 0.0
    for x in weights:
        total += float(x)
    n = len(weights)
    p = [float(x) * n / total for x in weights]
    alias = list(range(n))
    small = [i for i in range(n) if p[i] < 1.0]
    large = [i for i in range(n) if p[i] >= 1.0]
    while small and large:
        s, g = small.pop(), large.pop()
        alias[s] = g
        p[g] = (p[g] + p[s]) - 1.0
        (small if p[g] < 1.0 else large).append(g)
    thr = [int(p[i] * 2.0 ** 64) if alias[i] != i and p[i] < 1.0 else 2 ** 64 - 1 for i in range(n)]
    return thr, alias


M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    k0, k1 = key & M32, key >> 32 & M32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (p1 >> 32 & M32) ^ c1 ^ k0, p1 & M32, (p0 >> 32 & M32) ^ c3 ^ k1, p0 & M32
        k0, k1 = k0 + 0x9E3779B9 & M32, k1 + 0xBB67AE85 & M32
    return c0, c1, c2, c3


class _Walls:
    """Particles between two isothermal walls (periodic x and y) in 64 bits,
    all at once: the random words are the library's, the arithmetic torch's."""

    def __init__(self, mat, geo, n, key, fp64, t_max=None):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.n, self.key, self.fp64, self.t_max = n, key, fp64, t_max
        C = mat.C
        if C is None:
            x = 1.054571817e-34 * mat.omega / (1.380649e-23 * mat.T_lin)
            C = mat.D * (1.380649e-23 * (x / 2) ** 2 / np.sinh(x / 2) ** 2) * mat.domega
        self.C, self.bins = C, C.size
        self.sums = C.sum(), (C * mat.v).sum()
        v = mat.v * 1e-3
        self.v, self.lam = self.f(v), self.f(v * (mat.tau * 1e12))
        self.emit_table, self.relax_table = (self.table(w) for w in (C * mat.v, C / mat.tau))
        self.L = [x * 1e9 for x in geo.L]
        self.box, self.dT = geo.L, [geo.face_T[4] - geo.T_eq, geo.face_T[5] - geo.T_eq]
        A = geo.L[0] * geo.L[1]
        E = [0.25 * A * self.sums[1] * abs(d) * (t_max or 1.0) for d in self.dT]
        self.E_tot, self.split = sum(E), int(E[0] / sum(E) * 2.0 ** 32)

    def f(self, a):
        return torch.as_tensor(np.asarray(a, dtype=np.float64), device=self.dev)

    def table(self, w):
        thr, alias = _alias(w)
        return [torch.tensor(a, dtype=torch.int64, device=self.dev)
                for a in ([t >> 32 for t in thr], [t & M32 for t in thr], alias)]

    def uniform(self, w, add):
        return (w.double() + add) * 2.0 ** -32 if self.fp64 else ((w >> 8).double() + add) * 2.0 ** -24

    def flight(self, lo, hi):
        m = (hi << 21) ^ (lo >> 11) if self.fp64 else hi >> 8
        return -torch.log((m.double() + 1.0) * (2.0 ** -53 if self.fp64 else 2.0 ** -24))

    def pick(self, table, w, lo, hi):
        col = w * self.bins >> 32
        th, tl, alias = table[0][col], table[1][col], table[2][col]
        return torch.where((hi < th) | ((hi == th) & (lo < tl)), col, alias)

    def direction(self, mu, w):
        s, phi = torch.sqrt(torch.clamp(1.0 - mu * mu, min=0.0)), 2.0 * math.pi * self.uniform(w, 0.0)
        return torch.stack([s * torch.cos(phi), s * torch.sin(phi), mu])

    def emit(self):
        self.pid = torch.arange(self.n, dtype=torch.int64, device=self.dev)
        self.e = torch.zeros_like(self.pid)
        w0, w1, w2 = (_philox(self.pid, self.e, self.e, self.e + k, self.key) for k in range(3))
        hot = w1[3] < self.split
        sign = [1.0 if d > 0 else -1.0 for d in self.dT]
        self.s = torch.where(hot, sign[0], sign[1]).double()
        self.bin = self.pick(self.emit_table, w0[0], w0[1], w1[0])
        mu = torch.sqrt(self.uniform(w0[2], 1.0))
        self.u = self.direction(mu, w0[3])
        self.u[2] = torch.where(hot, mu, -mu)
        self.x = torch.stack([self.uniform(w2[0], 0.5) * self.L[0], self.uniform(w2[1], 0.5) * self.L[1],
                              torch.where(hot, 0.0, self.L[2]).double()])
        self.d = self.lam[self.bin] * self.flight(w1[1], w1[2])
        self.t = self.uniform(w2[3], 0.0) * self.t_max * 1e12 if self.t_max else torch.zeros_like(self.d)
        self.X = torch.zeros_like(self.d)

    def hit(self):
        """Distance to the nearest face and its axis (ties: lowest face)."""
        big = torch.full_like(self.d, 1e300)
        c = []
        for a, up in ((1, False), (0, True), (1, True), (0, False), (2, False), (2, True)):
            u = self.u[a]
            q = ((self.L[a] if up else 0.0) - self.x[a]) / u
            c.append(torch.where(u > 0 if up else u < 0, torch.clamp(q, min=0.0), big))
        d, face = torch.stack(c).min(0)
        return d, torch.tensor([1, 0, 1, 0, 2, 2], device=self.dev)[face], face

    def relax(self, i):
        w = _philox(self.pid[i], torch.zeros_like(i), self.e[i], torch.zeros_like(i), self.key)
        if self.fp64:
            w1 = _philox(self.pid[i], torch.zeros_like(i), self.e[i], torch.ones_like(i), self.key)
            b, free = self.pick(self.relax_table, w[0], w[1], w1[0]), self.flight(w1[1], w1[2])
        else:
            m = w[0] * self.bins
            col = m >> 32
            b = torch.where((m & M32) < self.relax_table[0][col], col, self.relax_table[2][col])
            free = self.flight(w[1], w[1])
        self.bin[i] = b
        self.d[i] = self.lam[b] * free
        self.u[:, i] = self.direction(1.0 - 2.0 * self.uniform(w[2], 1.0), w[3])

    def keep(self, m):
        for k in ("pid", "e", "s", "bin", "d", "t", "X"):
            setattr(self, k, getattr(self, k)[m])
        self.u, self.x = self.u[:, m], self.x[:, m]

    def trace(self, tally):
        """Steps every particle to its end; tally(seg, t_end) sees each flight."""
        self.emit()
        ev, top, end = 0, 0, {"X": 0.0, "X2": 0.0, "abs": 0.0, "n": 0}
        emitted = float(self.s.sum())
        while self.pid.numel():
            db, axis, face = self.hit()
            relax = self.d < db
            seg = torch.where(relax, self.d, db)
            fin = torch.zeros_like(relax)
            t_end = self.t + seg / self.v[self.bin]
            if self.t_max:
                left = (self.t_max * 1e12 - self.t) * self.v[self.bin]
                fin = (left <= self.d) & (left <= db)
                relax, seg = relax & ~fin, torch.where(fin, left, seg)
                t_end = torch.where(fin, self.t_max * 1e12, t_end)
            tally(seg, t_end, fin)
            self.X += self.s * seg * self.u[2]
            self.x += seg * self.u
            self.t = t_end
            self.e += (~fin).long()
            wall = ~relax & ~fin
            self.d = torch.where(wall, self.d - seg, self.d)
            for a in range(2):
                on = wall & (axis == a)
                low = (face == 0) | (face == 3)
                self.x[a] = torch.where(on, torch.where(low, self.L[a], 0.0).double(), self.x[a])
            i = relax.nonzero().flatten()
            if i.numel():
                self.relax(i)
            gone = wall & (axis == 2)
            done = gone | fin
            if bool(done.any()):
                X = self.X[done]
                end["X"] += float(X.sum())
                end["X2"] += float((X * X).sum())
                end["abs"] += float(self.s[gone].sum())
                end["n"] += int(gone.sum())
                ev += int((self.e[done] + 1).sum())
                top = max(top, int(self.e[done].max()) + 1)
                self.keep(~done)
        return ev, top, emitted, end


def _exact_slab(case, key):
    mat, geo = _slab_parts(case)
    w = _Walls(mat, geo, case["n"], key, case["fp64"])
    nc = case["cells"]
    part = torch.zeros(max(nc, 1), 4, dtype=torch.float64, device=w.dev)
    full = torch.zeros(nc + 2, 4, dtype=torch.float64, device=w.dev)
    qbin = torch.zeros(w.bins, dtype=torch.float64, device=w.dev)
    h = w.L[2] / max(nc, 1)

    def tally(seg, t_end, fin):
        uz = w.u[2]
        qbin.index_add_(0, w.bin, w.s * seg * uz)
        if not nc:
            return
        f = torch.stack([w.s / w.v[w.bin], w.s * w.u[0], w.s * w.u[1], w.s * uz], 1)
        a, b = w.x[2], w.x[2] + seg * uz
        lo, hi = torch.minimum(a, b), torch.maximum(a, b)
        i, j = (torch.clamp(torch.floor(z / h).long(), 0, nc - 1) for z in (lo, hi))
        one = (i == j).double()
        per = f / torch.abs(uz).clamp(min=1e-300)[:, None]
        first = torch.where(i == j, hi - lo, (i + 1) * h - lo)[:, None] * per
        flat = (uz == 0)[:, None]
        part.index_add_(0, i, torch.where(flat, f * seg[:, None], first))
        part.index_add_(0, j, torch.where(flat, 0.0 * f, (hi - j * h)[:, None] * per) * (1.0 - one)[:, None])
        run = per * h * (j > i + 1).double()[:, None]
        full.index_add_(0, i + 1, run)
        full.index_add_(0, j, -run)

    ev, top, emitted, end = w.trace(tally)
    V = geo.L[0] * geo.L[1] * geo.L[2]
    E = w.E_tot / case["n"]
    n, grad = case["n"], (w.dT[1] - w.dT[0]) / geo.L[2]
    q = E / V * end["X"] * 1e-9
    var = (end["X2"] - end["X"] ** 2 / n) / (n - 1)
    se = E / V * 1e-9 * math.sqrt(max(var, 0.0) * n)
    stats = [-q / grad, se / abs(grad), q, se, end["X"], end["X2"], ev, 0.0, w.E_tot, top, -q / grad, emitted,
             end["abs"], 0.0, n, end["n"]]
    res = {"stats": torch.tensor([stats], dtype=torch.float64), "T": None, "q": None, "q_bin": None}
    if nc:
        sums = (part + torch.cumsum(full, 0)[:nc]) * (E / (V / nc))
        res["T"] = (sums[:, 0] / w.sums[0] * 1e-12)[None]
        # with axis_flux the library keeps the axial flux alone
        keep = torch.tensor([0.0, 0.0, 1.0] if case["axis_flux"] and not case["fp64"] else [1.0] * 3, device=w.dev)
        res["q"] = (sums[:, 1:] * 1e-9 * keep)[None]
    if case["per_bin"]:
        res["q_bin"] = (E / V * qbin * 1e-9)[None]
    return res


def _exact_walls(case, key):
    mat, geo = _wall_parts()
    t = _wall_times(case)
    w = _Walls(mat, geo, case["n"], key, False, t_max=float(t[-1]))
    nc, times = case["cells"], w.f(t * 1e12)
    out = torch.zeros(len(t), nc, 4, dtype=torch.float64, device=w.dev)

    def tally(seg, t_end, fin):
        for m in range(len(t)):
            i = ((times[m] >= w.t) & ((times[m] < t_end) | fin)).nonzero().flatten()
            v = w.v[w.bin[i]]
            z = w.x[2][i] + v * (times[m] - w.t[i]) * w.u[2][i]
            c = torch.clamp(torch.floor(z * (nc / w.L[2])).long(), 0, nc - 1)
            s = w.s[i]
            out[m].index_add_(0, c, torch.stack([s] + [s * v * w.u[a][i] for a in range(3)], 1))

    ev, top, emitted, end = w.trace(tally)
    E = w.E_tot / case["n"]
    vc = geo.L[0] * geo.L[1] * geo.L[2] / nc
    out[..., 0] *= E / (w.sums[0] * vc)
    out[..., 1:] *= E / vc * 1e3
    stats = [0.0] * 6 + [ev, 0.0, w.E_tot, top, 0.0, emitted, end["abs"], 0.0, case["n"], end["n"]]
    return {"tally": out.reshape(len(t), nc, 1, 1, 4), "stats": torch.tensor(stats, dtype=torch.float64)}


def exact(case, seed):
    key = 1 + seed * 2654435761 % (1 << 40)
    # diffuse films, pores and the hot spot trace chains of up to a million
    # events, one after the other: too long for whole-array steps
    if case["kind"] == "slab" and work(case)["flops"] < 2e11:
        return _exact_slab(case, key)
    if case["kind"] == "walls":
        return _exact_walls(case, key)
    return None
