"""Edges of the FP32 steady run that its usual sizes do not reach.

* free paths so long that the summed tallies leave 64-bit fixed point: the
  run's sum is that of its particles;
* gradients of boxes without pore or walls whose periods do not fit one pass:
  the replay finds the forward pass's tallies;
* bin counts whose tables leave the tail 32 draw slots per warp, or no room for
  a table: the same bits as without the tail;
* bin counts whose tables leave a warp's batch 16 slots: the same bits in every
  launch shape.
"""
import numpy as np
import pytest

from inputs import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2104_03573_gb300 import _lib as L  # noqa: E402
from paper_2104_03573_gb300 import api  # noqa: E402


@pytest.mark.parametrize("mfp", [100e-9, 1e-4, 30.0])
@pytest.mark.parametrize("tail", [0, -1])
def test_sum_of_tallies_is_that_of_the_particles(mfp, tail):
    # 2e5 particles, each |X| of the order of the free path; fixed point holds
    # sums up to 2^43 nm = 8.8e3 m
    g = W.film(1.0, W=1.0)
    g.face_type = [W.PERIODIC] * 6
    cfg = api.SteadyConfig(seed=7, precision=L.FP32_TRACE, n_scat_max=3, tally_axis=1, max_events=10 ** 7,
                           tail_lanes=tail)
    o = api.run_steady(api.Material(W.gray(6000.0, mfp)), [api.Geometry(g)], [200_000], cfg, per_particle=True)
    torch.cuda.synchronize()
    X = o.X_pp.cpu().numpy()
    # exact whole numbers per block, rounded when a block adds: 1e3 additions at
    # most, each within 2^-53 of the sum of magnitudes
    for k, ref, mag in ((L.STAT_SUMX, X.sum(), np.abs(X).sum()), (L.STAT_SUMX2, (X * X).sum(), (X * X).sum())):
        assert abs(o.stats[0, k].item() - ref) < 1e-12 * mag


@pytest.mark.parametrize("tail", [0, -1])
@pytest.mark.parametrize("axis,n", [(0, 17), (1, 17), (2, 17), (1, 40)])
def test_two_pass_gradient_of_a_film(axis, n, tail):
    # the film's walls across `axis`, the control gradient along it: the other
    # two axes are periodic, and forward flights alone would run through them
    ft, fp = [W.PERIODIC] * 6, [0.0] * 6
    for f in {0: (W.FACE_X0, W.FACE_XL), 1: (W.FACE_Y0, W.FACE_YL), 2: (W.FACE_Z0, W.FACE_ZL)}[axis]:
        ft[f], fp[f] = W.ADIABATIC, 0.3
    size, grad = [100e-9] * 3, [0.0] * 3
    size[axis] = 300e-9
    grad[(axis + 1) % 3] = -1e6
    g = W.Geometry(L=size, face_type=ft, face_p=fp, grad_T=tuple(grad))
    cfg = api.SteadyConfig(seed=5, precision=L.FP32_TRACE, n_scat_max=n, tally_axis=(axis + 1) % 3, per_bin=True,
                           max_events=10 ** 7, tail_lanes=tail)
    M, G = api.Material(W.bvk_holland()), api.Geometry(g)
    fwd, go = api.grad(M, G, 20_011, cfg)
    torch.cuda.synchronize()
    assert fwd.stats[0, L.STAT_STATUS].item() == 0 and fwd.stats[0, L.STAT_N].item() == 20_011
    # a run without gradient takes whole flights: other roundings of the
    # positions, which a few long trajectories turn into other events
    run = api.run_steady(M, [G], [20_011], cfg)
    torch.cuda.synchronize()
    k, s = L.STAT_KAPPA, L.STAT_KAPPA_SE
    assert abs(fwd.stats[0, k].item() - run.stats[0, k].item()) < 3 * run.stats[0, s].item()
    assert torch.isfinite(go.dkappa_dlogtau).all()


# with the per-bin flux: 4110 bins leave a gradient 32 slots, 5100 a forward
# run; at 6300 and 12 600 the flux, and the per-bin constants, are in global memory
@pytest.mark.parametrize("bins", [4110, 5100, 6300, 12_600])
@pytest.mark.parametrize("kind", ["film", "pore", "walls", "batch"])
def test_tails_at_bin_counts_between(kind, bins):
    M = api.Material(W.bvk_holland(n_per_branch=bins // 3))
    assert M.n_bins == bins
    gs = {"film": [W.film(100e-9, p=0.4)], "pore": [W.pore_lattice(100e-9, 0.25, 200e-9, p_pore=0.4)],
          "walls": [W.nanomesh(p_pore=0.4)], "batch": [W.film(30e-9), W.film(2000e-9), W.film(200e-9)]}[kind]
    outs = []
    for tail in (-1, 8):
        cfg = api.SteadyConfig(seed=45, precision=L.FP32_TRACE, tally_axis=1, n_scat_max=10, per_bin=True,
                               max_events=10 ** 6, tail_lanes=tail)
        o = api.run_steady(M, [api.Geometry(g) for g in gs], [5003] * len(gs), cfg, per_particle=True)
        torch.cuda.synchronize()
        outs.append([getattr(o, k).cpu().numpy() for k in ("events_pp", "X_pp", "q_bin")])
    for a, b in zip(*outs):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("bins", [4110, 5100, 6300, 12_600])
@pytest.mark.parametrize("p", [0.0, 0.4])
def test_gradient_tails_at_bin_counts_between(p, bins):
    M = api.Material(W.bvk_holland(n_per_branch=bins // 3))
    G = api.Geometry(W.pore_lattice(100e-9, 0.25, 200e-9, p_pore=p))
    outs = []
    for tail in (-1, 8):
        cfg = api.SteadyConfig(seed=46, precision=L.FP32_TRACE, tally_axis=1, n_scat_max=10, per_bin=True,
                               max_events=10 ** 6, tail_lanes=tail)
        fwd, go = api.grad(M, G, 5003, cfg)
        torch.cuda.synchronize()
        assert fwd.stats[0, L.STAT_N].item() == 5003
        outs.append([t.cpu().numpy() for t in (fwd.q_bin, go.dkappa_dlogtau, go.dkappa_dp)])
    # the same particles: whole-number sums equal, FP64 sums over particles in another order
    assert np.array_equal(outs[0][0], outs[1][0])
    for a, b in zip(outs[0][1:], outs[1][1:]):
        assert np.max(np.abs(a - b)) < 1e-9 * np.max(np.abs(a))


# with per-bin flux 4800 bins leave blocks of 768 threads 32 slots, 5010 16;
# without it 5850 and 6390
@pytest.mark.parametrize("bins,per_bin", [(4800, True), (5010, True), (5850, False), (6390, False)])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("n", [1, 33, 20_011])
def test_batches_at_bin_counts_between(n, walls, bins, per_bin):
    M = api.Material(W.bvk_holland(n_per_branch=bins // 3))
    G = api.Geometry(W.nanomesh(p_pore=0.4) if walls else W.slab_z(1e-6, 300.5, 299.5, lateral=1e-6))
    base = None
    for threads in (256, 512, 768, 1024):
        cfg = api.SteadyConfig(seed=47, precision=L.FP32_TRACE, tally_axis=1 if walls else 2, n_cells=33, cell_axis=2,
                               n_scat_max=10 if walls else 0, per_bin=per_bin, max_events=10 ** 6,
                               threads_per_block=threads)
        o = api.run_steady(M, [G], [n], cfg, per_particle=True)
        torch.cuda.synchronize()
        assert o.stats[0, L.STAT_N].item() == n
        cur = [getattr(o, k).cpu().numpy() for k in ("events_pp", "X_pp", "T", "q") + (("q_bin",) if per_bin else ())]
        base = base or cur
        for a, b in zip(base, cur):
            assert np.array_equal(a, b), threads
