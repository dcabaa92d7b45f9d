"""The CTA bins at the edges of their size ranges, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_1503_04500_gb300 import inputs as gen
from parity_check import check_fp32_every_column
from test_gpu_parity import assert_fp64_parity, gpu_M

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
rsai = pytest.importorskip("paper_1503_04500_gb300.rsai")


@pytest.mark.parametrize("precision", ["fp64", "fp32_refine"])
@pytest.mark.parametrize("N, eps, drop", [(9, 0.1, "adaptive"), (10, 0.12, "none")])
def test_columns_between_the_warp_and_the_large_cta_bin(precision, N, eps, drop):
    """Columns with 32 < |J| <= 64 (one small CTA each) and, in the first problem, some
    with more, which move on to the next bin; the frozen pattern's refit takes the same bins."""
    A = gen.convdiff3d(N)
    kw = dict(c=3, l_max=15, eps=eps, tol=1e-3, drop=drop)
    h, dA, res, rho, loops, flags, st = gpu_M(A, precision=precision, **kw)
    ref = oracle.build(A, **kw)
    sizes = np.diff(ref.colptr)
    assert (sizes > 32).sum() > 100 and (drop == "none" or (sizes > 64).sum() > 50)
    assert st["cols_bin"][1] > 0 and st["n_failed"] == 0
    if precision == "fp64":
        assert_fp64_parity(A, ref, res, rho, loops, flags, st)
    else:
        check_fp32_every_column(A, res, rho, ref)
    mv, rho2 = h.refit(dA.val)
    tol = 1e-9 if precision == "fp64" else 1e-6
    np.testing.assert_allclose(mv.cpu().numpy(), res[2], rtol=tol, atol=tol * np.abs(res[2]).max())
    np.testing.assert_allclose(np.sqrt(rho2.cpu().numpy()), rho, rtol=tol, atol=1e-12)
