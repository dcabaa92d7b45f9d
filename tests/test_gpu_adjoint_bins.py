"""The adjoint in the CTA bins where its index sets change form."""
import numpy as np
import pytest

from paper_1503_04500_gb300 import inputs as gen
from test_gpu_cta_bins import embedded

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
rsai = pytest.importorskip("paper_1503_04500_gb300.rsai")


@pytest.mark.parametrize("precision", ["fp64", "fp32_refine"])
def test_adjoint_of_large_problems(precision):
    """Products with A(I,J) look indices up in a bitmap of n bits while it fits shared memory (n up
    to about 1.2 million) and search the sorted sets beyond, in the same order of every
    sum: the block's gradient is the small problem's bit for bit.  Rows of M longer
    than 64 entries, which a whole warp takes, are among them."""
    block = gen.powerlaw(900, seed=5, dmax=100)
    kw = dict(c=5, l_max=8, eps=0.4, tol=1e-3, drop="fixed", precision=precision)
    grads = []
    for A in (block, embedded(block, 1_300_000)):
        dA = rsai.DeviceMatrix.from_host(A)
        h = rsai.build(dA, **kw)
        assert h.stats()["cols_bin"][2] > 0
        rp = h.M()[0]
        nnz = int(rp[-1])
        longest = int((rp[1:] - rp[:-1]).max())
        assert longest > 64
        m = int(rp[block.n])  # entries of M in the block's rows
        gM = torch.zeros(nnz, dtype=torch.float64, device="cuda")
        gM[:m] = torch.sin(torch.arange(m, dtype=torch.float64, device="cuda"))
        gr = torch.zeros(A.n, dtype=torch.float64, device="cuda")
        gr[: block.n] = torch.linspace(-1, 1, block.n, dtype=torch.float64, device="cuda")
        g = h.backward(dA.val, gM, gr)
        grads.append(g[: block.nnz].cpu().numpy())
        h.free()
    assert np.abs(grads[0]).max() > 0
    assert np.array_equal(grads[0], grads[1])
