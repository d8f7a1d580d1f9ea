"""Runs in which lanes trace several particles one after the other.

* FP64 kernels at the edges of their distribution of particles: equal shares
  per warp (up to 32 particles on each of four warps per SM), chunks of 32
  preassigned to six warps per SM, the first one from the work counter, and
  several per lane; steady runs, transients and both gradient estimators equal
  the oracle's (per particle in every bit, tallies, which are sums of atomics,
  within 1e-9 of their largest magnitude);
* the transient at full size in windows of ten measurement times equals the
  run in one window in every bit.
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
SMS = torch.cuda.get_device_properties(0).multi_processor_count
SHARES, CHUNKS = 32 * 4 * SMS, 32 * 6 * SMS
EDGES = {"shares": SHARES, "shares+1": SHARES + 1, "chunks": CHUNKS, "chunks+1": CHUNKS + 1, "several": 2 * CHUNKS + 5}


def _close(got, ref, what):
    ok, err = rel_close(np.asarray(got).reshape(np.shape(ref)), ref, RTOL)
    assert ok, (what, err)


@pytest.mark.parametrize("n", EDGES.values(), ids=EDGES.keys())
def test_fp64_steady_refills(n):
    wl = W.si_slab_c2(n=n)
    mat, g, run = wl.material, wl.geometries[0], replace(wl.run, n_cells=7)
    gg = gpu_steady(mat, [g], [n], run, L.FP64_PLAIN, per_particle=True)
    ref = oracle.run_steady(mat, g, run, per_particle=True)
    assert gg["stats"][0][L.STAT_N] == n
    assert np.array_equal(gg["events_pp"], ref["events_pp"])
    assert np.array_equal(gg["X_pp"], ref["X_pp"])
    for k in ("T", "q", "q_bin"):
        _close(gg[k][0], ref[k], k)


@pytest.mark.parametrize("n", EDGES.values(), ids=EDGES.keys())
@pytest.mark.parametrize("average", [False, True])
@pytest.mark.parametrize("regions", [False, True])
@pytest.mark.parametrize("walls", [False, True])
def test_fp64_transient_refills(walls, regions, average, n):
    # 20 ps: a few events per particle; a hot spot at the start, or walls that
    # emit over the whole time (a lane's next particle may start before its last)
    wl = W.ballistic_transient_e1(n=n) if walls else W.transient_box_c3(n=n, grid=(4, 3, 5), n_times=6)
    mat, g, run = W.bvk_holland(), wl.geometries[0], wl.run
    run.t_max, run.time_average = 2e-11, average
    if regions:
        x, y, z = g.L
        run.regions = [((0.2 * x, 0.9 * x, 0.1 * y, 0.8 * y, 0.0, 0.7 * z), (2, 3, 1)), ((0.0, x, 0.0, y, 0.0, z), (1, 2, 2))]
    run.t_meas = run.t_max * np.arange(1, 7) / 6
    gg = gpu_transient(mat, g, run, L.FP64_PLAIN, per_particle=True)
    ref = oracle.run_transient(mat, g, run, per_particle=True)
    assert gg["stats"][L.STAT_N] == n
    assert np.array_equal(gg["events_pp"], ref["events_pp"])
    for s in (slice(0, 1), slice(1, 4)):
        _close(gg["tally"][..., s], ref["tally"][..., s], s)


@pytest.mark.parametrize("n", EDGES.values(), ids=EDGES.keys())
@pytest.mark.parametrize("est", [L.DP_LIKELIHOOD_RATIO, L.DP_MEASURE_VALUED])
def test_fp64_gradient_refills(est, n):
    # a lane's next particle comes after a phantom trace (measure-valued): its
    # tallies are bound again and its period list starts anew
    wl = W.pore_film_c5(n=n, p_pore=0.3)
    mat, g = wl.material, wl.geometries[0]
    run = replace(wl.run, n_cells=5, n_scat_max=2, max_events=200)
    rng = np.random.default_rng(9)
    dirs = rng.normal(size=(1, mat.n_bins))
    cfg = api.SteadyConfig(seed=run.seed, precision=L.FP64_PLAIN, n_scat_max=2, max_events=200, n_cells=5,
                           cell_axis=run.cell_axis, tally_axis=run.tally_axis, per_bin=True)
    fwd = api.SteadyOutputs(1, mat.n_bins, 5, True, n, per_particle=True)
    fwd, go = api.grad(api.Material(mat), api.Geometry(g), n, cfg, dirs=dirs, fwd=fwd, dp_estimator=est)
    torch.cuda.synchronize()
    ref = oracle.run_steady(mat, g, run, per_particle=True, grad=True, dirs=dirs, dp_estimator=est)
    assert fwd.stats[0, L.STAT_N].item() == n
    assert np.array_equal(fwd.events_pp.cpu().numpy().astype(np.uint32), ref["events_pp"])
    assert np.array_equal(fwd.X_pp.cpu().numpy(), ref["X_pp"])
    for k in ("T", "q", "q_bin"):
        _close(getattr(fwd, k)[0].cpu().numpy(), ref[k], k)
    _close(go.dkappa_dlogtau.cpu().numpy(), ref["dkappa_dlogtau"], "dlogtau")
    _close(go.dkappa_dir[:1, 0].cpu().numpy(), ref["dkappa_dir"], "dir")
    assert go.dkappa_dp[0].item() == pytest.approx(ref["dkappa_dp"], rel=RTOL)


def test_transient_full_size_in_windows_of_ten_times():
    wl = W.transient_box_c3()                             # 1e8 particles, 64x64x32 cells x 200 times
    mat, geo, run = wl.material, wl.geometries[0], wl.run
    M, G = api.Material(mat), api.Geometry(geo)
    outs = []
    for wt in (10, len(run.t_meas)):
        out = api.TransientOutputs(len(run.t_meas), run.grid, run.n)
        cfg = api.TransientConfig(seed=run.seed, t_max=run.t_max, t_meas=run.t_meas, grid=run.grid,
                                  precision=L.FP32_TRACE, window_times=wt)
        api.run_transient(M, G, run.n, cfg, out=out)
        torch.cuda.synchronize()
        st = out.stats.cpu().numpy()
        assert st[L.STAT_STATUS] == 0 and st[L.STAT_N] == run.n
        outs.append(out)
    assert torch.equal(outs[0].tally, outs[1].tally)
    assert torch.equal(outs[0].stats, outs[1].stats)
