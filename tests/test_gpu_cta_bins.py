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


def embedded(block, n):
    """diag(block, I): the block's columns are built as in the block alone."""
    m = block.n
    rows = np.concatenate([np.repeat(np.arange(m), np.diff(block.row_ptr)), np.arange(m, n)])
    cols = np.concatenate([block.col_idx, np.arange(m, n)])
    return gen.from_coo(n, rows, cols, np.concatenate([block.val, np.ones(n - m)]))


@pytest.mark.parametrize("precision", ["fp64", "fp32_refine"])
@pytest.mark.parametrize("n", [1_200_000, 1_300_000])
def test_index_sets_of_large_problems(precision, n):
    """The global bin keeps index sets as bitmaps of n bits while they fit its shared memory
    (n up to about 1.2 million) and sorts and searches beyond; both give the small problem's
    columns bit for bit."""
    block = gen.powerlaw(900, seed=5, dmax=100)
    kw = dict(c=5, l_max=8, eps=0.4, tol=1e-3, drop="fixed")
    _, _, small, rho_s, loops_s, _, st = gpu_M(block, precision=precision, **kw)
    assert st["cols_bin"][2] > 0
    _, _, large, rho, loops, _, _ = gpu_M(embedded(block, n), precision=precision, **kw)
    m, nnz = block.n, small[0][-1]
    assert np.array_equal(large[0][: m + 1], small[0])
    assert np.array_equal(large[1][:nnz], small[1]) and np.array_equal(large[2][:nnz], small[2])
    assert np.array_equal(rho[:m], rho_s) and np.array_equal(loops[:m], loops_s)
