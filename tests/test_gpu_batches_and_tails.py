"""Edges of the tracers' batches, table builds, snapshot records and tails.

* alias tables at the edges of the builder's runs per thread, of its 32-lane
  scan and of its shared-memory range: equal to the oracle's in every bit;
* FP64 runs of particle counts around whole batches of 32 per warp and one
  warp per SM: every particle the oracle's, tallies (sums of atomics over
  copies) within 1e-9 of their largest magnitude, also where the copies of the
  sums do not fit the workspace;
* FP32 runs of few particles: the same bits for every launch shape;
* snapshots added as whole records in one window: the oracle's in FP64, and in
  FP32 the same integers as in windows of one measurement time;
* the tail's event loops along every axis, with diffuse, specular and mixed
  walls: the same bits as without the tail.
"""
from dataclasses import replace

import numpy as np
import pytest

import oracle
from inputs import workloads as W
from gpu_helpers import gpu_steady, gpu_transient, rel_close

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2104_03573_gb300 import _lib as L  # noqa: E402
from paper_2104_03573_gb300 import api  # noqa: E402

RTOL = 1e-9
# faces of each axis (lower, upper)
FACES = {0: (W.FACE_X0, W.FACE_XL), 1: (W.FACE_Y0, W.FACE_YL), 2: (W.FACE_Z0, W.FACE_ZL)}


def _weights(kind, n, rng):
    if kind == "equal":
        return np.full(n, 1e3)
    C = rng.exponential(size=n) * 1e3
    if kind == "one_bin":          # every small bin takes the same large one
        C[:] = 1e-3
        C[n // 2] = 1e6
    if kind == "zeros":
        C[rng.uniform(size=n) < 0.5] = 0.0
        C[0] = 1.0
    return C


@pytest.mark.parametrize("kind", ["random", "equal", "one_bin", "zeros"])
@pytest.mark.parametrize("n", [1, 2, 7, 8, 31, 33, 255, 257, 9216, 9217])
def test_alias_tables_equal_the_oracles(n, kind):
    rng = np.random.default_rng(n)
    m = W.Material(omega=np.linspace(1e12, 7e13, n), v=rng.uniform(1e3, 9e3, n), tau=10 ** rng.uniform(-12, -9, n),
                   C=_weights(kind, n, rng), T_lin=300.0)
    t_g, t_o = api.Material(m).tables(), oracle.tables(m)
    for k in ("C", "alias", "thr", "prob"):
        assert np.array_equal(t_g[k], t_o[k]), k
    assert t_g["sum_Cv"] == t_o["sum_Cv"] and t_g["C_tot"] == t_o["C_tot"]


# 152 SMs: one warp each takes 4864 particles at once
@pytest.mark.parametrize("n", [1, 32, 33, 4864, 4865, 20_001])
@pytest.mark.parametrize("cells", [0, 7])
def test_fp64_runs_around_whole_batches(n, cells):
    wl = W.si_slab_c2(n=n)
    mat, g, run = wl.material, wl.geometries[0], replace(wl.run, n_cells=cells)
    gg = gpu_steady(mat, [g], [n], run, L.FP64_PLAIN, per_particle=True)
    ref = oracle.run_steady(mat, g, run, per_particle=True)
    assert np.array_equal(gg["events_pp"], ref["events_pp"])
    assert np.array_equal(gg["X_pp"], ref["X_pp"])
    for k in ("T", "q", "q_bin") if cells else ("q_bin",):
        ok, err = rel_close(gg[k][0].reshape(ref[k].shape), ref[k], RTOL)
        assert ok, (k, err)
    assert gg["stats"][0][L.STAT_N] == n


def test_fp64_sums_in_a_workspace_without_room_for_their_copies():
    wl = W.si_slab_c2(n=5000)
    mat, g, run = wl.material, wl.geometries[0], wl.run
    M, G = api.Material(mat), api.Geometry(g)
    cfg = api.SteadyConfig(seed=run.seed, precision=L.FP64_PLAIN, n_cells=run.n_cells, tally_axis=2, per_bin=True)
    ws = torch.zeros(api.steady_workspace_size(M, [G], [run.n], cfg), dtype=torch.uint8, device="cuda")
    a = api.run_steady(M, [G], [run.n], cfg, workspace=ws)
    b = api.run_steady(M, [G], [run.n], cfg, workspace=ws[:-256])
    torch.cuda.synchronize()
    for k in ("T", "q", "q_bin"):
        ok, err = rel_close(getattr(b, k).cpu().numpy(), getattr(a, k).cpu().numpy(), RTOL)
        assert ok, (k, err)


@pytest.mark.parametrize("n", [1, 31, 33, 4097])
def test_fp32_small_runs_keep_their_bits_in_every_launch_shape(n):
    wl = W.si_slab_c2(n=n)
    M, G = api.Material(wl.material), api.Geometry(wl.geometries[0])
    base = None
    for threads, refill in ((0, 0), (256, 1), (1024, 32)):
        cfg = api.SteadyConfig(seed=7, precision=L.FP32_TRACE, n_cells=33, tally_axis=2, per_bin=True,
                               threads_per_block=threads, refill_threshold=refill)
        o = api.run_steady(M, [G], [n], cfg, per_particle=True)
        torch.cuda.synchronize()
        cur = {k: getattr(o, k).cpu().numpy() for k in ("events_pp", "X_pp", "T", "q", "q_bin")}
        assert o.stats[0, L.STAT_N].item() == n
        base = base or cur
        for k in cur:
            assert np.array_equal(cur[k], base[k]), (threads, refill, k)


@pytest.mark.parametrize("n,grid,times", [(1, (1, 1, 3), 2), (33, (5, 3, 7), 11), (4097, (3, 1, 2), 33)])
@pytest.mark.parametrize("even", [True, False])
def test_snapshot_records_on_ragged_grids(n, grid, times, even):
    wl = W.transient_box_c3(n=n, grid=grid, n_times=times)
    mat, g, run = wl.material, wl.geometries[0], wl.run
    if not even:
        run.t_meas = run.t_max * (np.arange(1, times + 1) / times) ** 2
    gg = gpu_transient(mat, g, run, L.FP64_PLAIN, per_particle=True)
    ref = oracle.run_transient(mat, g, run, per_particle=True)
    assert np.array_equal(gg["events_pp"], ref["events_pp"])
    for s in (slice(0, 1), slice(1, 4)):
        ok, err = rel_close(gg["tally"][..., s], ref["tally"][..., s], RTOL)
        assert ok, err
    a, b = (gpu_transient(mat, g, run, L.FP32_TRACE, per_particle=True, window_times=w) for w in (0, 1))
    assert np.array_equal(a["tally"], b["tally"]) and np.array_equal(a["events_pp"], b["events_pp"])


def _film_across(axis, p, wall, d):
    ft, fp, fT = [W.PERIODIC] * 6, [0.0] * 6, [0.0] * 6
    for f, dT in zip(FACES[axis], (0.5, -0.5)):
        ft[f], fp[f], fT[f] = wall, p, 300.0 + dT
    size, grad = [100e-9] * 3, [0.0] * 3
    size[axis] = d
    tally = axis
    if wall == W.ADIABATIC:
        tally = (axis + 1) % 3
        grad[tally] = -1e6
    return W.Geometry(L=size, face_type=ft, face_p=fp, face_T=fT, grad_T=tuple(grad)), tally


def _same_with_and_without_tail(mat, geo, n, tally, **kw):
    M, G = api.Material(mat), api.Geometry(geo)
    outs = []
    for tail in (-1, 8):
        cfg = api.SteadyConfig(seed=45, precision=L.FP32_TRACE, tally_axis=tally, n_scat_max=10,
                               max_events=kw.get("max_events", 10 ** 7), n_cells=kw.get("cells", 0), per_bin=True,
                               tail_lanes=tail)
        o = api.run_steady(M, [G], [n], cfg, per_particle=True)
        torch.cuda.synchronize()
        outs.append([getattr(o, k).cpu().numpy() for k in ("events_pp", "X_pp", "q_bin", "T", "q")
                     if getattr(o, k) is not None])
    for a, b in zip(*outs):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("p", [0.0, 0.4, 1.0])
@pytest.mark.parametrize("max_events", [10 ** 7, 777])
@pytest.mark.parametrize("d", [20e-9, 300e-9, 2000e-9])   # the period is 100 nm: few, several, many faces a flight
def test_film_tails_along_every_axis(axis, p, max_events, d):
    geo, tally = _film_across(axis, p, W.ADIABATIC, d)
    _same_with_and_without_tail(W.bvk_holland(), geo, 20_011, tally, max_events=max_events)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("d", [400e-9, 2000e-9])
def test_wall_to_wall_tails_along_every_axis(axis, d):
    geo, tally = _film_across(axis, 0.0, W.ISOTHERMAL, d)
    _same_with_and_without_tail(W.gray(6000.0, 5e-9), geo, 5003, tally)


@pytest.mark.parametrize("p", [0.0, 0.4, 1.0])
@pytest.mark.parametrize("cells", [0, 11])
def test_pore_and_wall_tails(p, cells):
    _same_with_and_without_tail(W.bvk_holland(), W.pore_lattice(100e-9, 0.25, 200e-9, p_pore=p, p_faces=p), 20_011, 1,
                                cells=cells)
    _same_with_and_without_tail(W.bvk_holland(), W.nanomesh(p_pore=p), 5003, 1, cells=cells)
