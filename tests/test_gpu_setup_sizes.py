"""The offsets of M at the edges of the scan's block counts."""
import numpy as np
import pytest

from paper_1503_04500_gb300 import inputs as gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
rsai = pytest.importorskip("paper_1503_04500_gb300.rsai")


@pytest.mark.parametrize("n", [1, 2, 1023, 1024, 1025, 32 * 1024, 4096 * 1024, 4096 * 1024 + 1])
def test_offsets_of_m_at_scan_edges(n):
    """M of a diagonal matrix: one entry per row, for every split of the scan into
    blocks of 1024 counts (folded up to 4096 blocks, three passes above)."""
    d = 2.0 ** (np.arange(n) % 5)
    i = np.arange(n)
    A = gen.from_coo(n, i, i, d)
    h = rsai.build(rsai.DeviceMatrix.from_host(A), c=3, l_max=2, eps=0.3, drop="none")
    rp, ci, va = h.M()
    assert torch.equal(rp, torch.arange(n + 1, device="cuda"))
    assert torch.equal(ci, torch.arange(n, dtype=torch.int32, device="cuda"))
    assert torch.equal(va, torch.as_tensor(1.0 / d, device="cuda"))
    h.free()
