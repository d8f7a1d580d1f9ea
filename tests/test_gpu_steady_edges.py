"""Edges of the FP32 steady run that its usual sizes do not reach.

* free paths so long that the summed tallies leave 64-bit fixed point: the
  run's sum is that of its particles.
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
