"""A handle with a column that outgrew every bin: the passes on its pattern report the failure
and take no room, in their pools of index sets, from that column."""
import numpy as np
import pytest

from paper_1503_04500_gb300 import inputs as gen
from test_gpu_failures import FailingAllocator

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
rsai = pytest.importorskip("paper_1503_04500_gb300.rsai")

RSAI_ERR_WORKSPACE, RSAI_COL_FAILED = 9, 8


class Recording(FailingAllocator):
    """Keeps the size of every request."""

    class Live(dict):
        def __init__(self):
            super().__init__()
            self.sizes = []

        def __setitem__(self, ptr, nbytes):
            self.sizes.append(nbytes)
            super().__setitem__(ptr, nbytes)

    def __init__(self):
        super().__init__()
        self.live = self.Live()


@pytest.mark.parametrize("precision", ["fp64", "fp32_refine"])
def test_passes_on_a_pattern_with_a_failed_column(precision):
    """Column 0 starts from a pattern of 4150 indices (the largest bin takes 4096); every other
    column of A is diagonal, so |I_k| = 1."""
    n, m = 4200, 4150
    i = np.arange(n)
    A = gen.from_coo(n, np.concatenate([i, i[1:m]]), np.concatenate([i, 0 * i[1:m]]),
                     np.concatenate([np.full(n, 2.0), np.full(m - 1, 0.25)]))
    dA = rsai.DeviceMatrix.from_host(A)
    # memory that the handle's buffers may come from holds no zeros
    torch.cuda.empty_cache()
    old = [torch.full((s,), 0x7F, dtype=torch.uint8, device="cuda") for s in [1 << 19] * 8 + [1 << 20] * 8 + [1 << 23] * 4]
    del old
    with Recording() as fa:
        h = rsai.build(dA, precision=precision, c=3, l_max=4, eps=0.3, drop="none", init="A", allow_failed=True)
        lib = rsai.load()
        _, loops, flags = (t.cpu().numpy() for t in h.columns())
        assert loops[0] == 0 and flags[0] & RSAI_COL_FAILED and not np.any(flags[1:] & RSAI_COL_FAILED)
        nnz = int(h.M()[0][-1])
        assert nnz == n - 1
        g = torch.empty(A.nnz, dtype=torch.float64, device="cuda")
        ones = torch.ones(nnz, dtype=torch.float64, device="cuda")
        stream = torch.cuda.current_stream().cuda_stream
        before = len(fa.live.sizes)
        status = lib.rsai_backward(h._h, dA.val.data_ptr(), ones.data_ptr(), None, g.data_ptr(), stream)
        assert status == RSAI_ERR_WORKSPACE
        asked = fa.live.sizes[before:]
        assert asked.count(8 * (n - 1)) >= 2 and 4 * (n - 1) in asked, asked  # r, w and I of the other columns
        assert max(asked) <= 8 * (A.nnz + n)
        with pytest.raises(rsai.RSAIError) as e:
            h.refit(dA.val)
        assert e.value.status == RSAI_ERR_WORKSPACE
        torch.cuda.synchronize()
        h.free()
