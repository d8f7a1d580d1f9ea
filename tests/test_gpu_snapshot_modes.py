"""The ways FP32 grid snapshots are added (whole records, word by word, by the
step) give the same integers: a window's slice of the tally decides, so the same
run in other windows takes another way."""
import numpy as np
import pytest

from inputs import workloads as W
from gpu_helpers import gpu_transient

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2104_03573_gb300 import _lib as L  # noqa: E402


# 6.6 MB in one window: word by word; 5 times a window are 0.33 MB: records.
# 210 MB and 839 MB are beyond the L2: by the step's count (few and many
# snapshots a step); 10 times a window are 42 MB: word by word.
@pytest.mark.parametrize("grid,times,windows", [((16, 16, 8), 100, (0, 50, 5)), ((64, 64, 32), 50, (0, 10)),
                                                ((64, 64, 32), 200, (0, 10))])
@pytest.mark.parametrize("n", [33, 100_003])
def test_snapshots_are_the_same_integers_in_every_mode(n, grid, times, windows):
    wl = W.transient_box_c3(n=n, grid=grid, n_times=times)
    base = None
    for w in windows:
        r = gpu_transient(wl.material, wl.geometries[0], wl.run, L.FP32_TRACE, per_particle=True, window_times=w)
        assert r["stats"][L.STAT_N] == n and r["stats"][L.STAT_STATUS] == 0
        base = base or r
        assert np.array_equal(r["tally"], base["tally"])
        assert np.array_equal(r["events_pp"], base["events_pp"])
        assert np.array_equal(r["stats"], base["stats"])


def test_walls_that_absorb_count_the_same_in_every_mode():
    # emission over the whole time and absorption: the lanes' counters
    wl = W.ballistic_transient_e1(n=50_001)
    a = gpu_transient(wl.material, wl.geometries[0], wl.run, L.FP32_TRACE, per_particle=True)
    b = gpu_transient(wl.material, wl.geometries[0], wl.run, L.FP32_TRACE, per_particle=True, threads_per_block=256)
    assert np.array_equal(a["tally"], b["tally"]) and np.array_equal(a["stats"], b["stats"])
    ev = a["events_pp"].astype(np.int64)
    assert a["stats"][L.STAT_EVENTS] == ev.sum() and a["stats"][L.STAT_MAX_EVENTS] == ev.max()
    assert 0 < a["stats"][L.STAT_ABSORBED] < 50_001
