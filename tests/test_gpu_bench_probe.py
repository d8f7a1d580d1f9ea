"""The bench's record probe adds what it says: whole records, every word alike."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("groups", [1, 255, 100_003])
def test_record_probe_adds_exactly(groups):
    import bench
    slots = torch.zeros(4096, dtype=torch.int64, device="cuda")
    other = torch.zeros_like(slots)
    s = torch.cuda.current_stream()
    probe = bench.load_probe()
    assert probe.bench_l2_record_probe(slots.data_ptr(), 4096, groups, ctypes.c_void_p(s.cuda_stream)) == 0
    assert probe.bench_l2_reduction_probe(other.data_ptr(), 4096, groups, ctypes.c_void_p(s.cuda_stream)) == 0
    torch.cuda.synchronize()
    assert int(slots.sum().item()) == 4 * groups
    assert torch.equal(slots, other)
