"""Columns of thousands of rows in the global bin: panels of fewer than kPanel columns (all that the
staging area takes of so many rows), single reflectors between them, and updates of a few or of many
appended columns."""
import numpy as np
import pytest

import oracle
from paper_1503_04500_gb300 import inputs as gen
from parity_check import check_fp32_every_column
from test_gpu_parity import assert_fp64_parity, gpu_M

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
rsai = pytest.importorskip("paper_1503_04500_gb300.rsai")


def long_columns(n, dense, fill, seed):
    """`dense` columns with about `fill` of all rows each; the others hold their diagonal entry only."""
    rng = np.random.default_rng(seed)
    i = np.arange(n)
    rows, cols, vals = [i], [i], [60.0 + rng.random(n)]
    for j in rng.choice(n, dense, replace=False):
        r = np.flatnonzero(rng.random(n) < fill)
        r = r[r != j]
        rows.append(r)
        cols.append(np.full(r.size, j))
        vals.append(rng.standard_normal(r.size))
    return gen.from_coo(n, *(np.concatenate(x) for x in (rows, cols, vals)))


# n rows of which FP64 panels of 16, 9, 4 or 3 columns fit the staging area (FP32: 16, 16, 9, 7);
# c appended columns and more per loop; the entries of A(:,J) stay within the bin's 131072
@pytest.mark.parametrize("n, dense, fill", [(1500, 40, 0.9), (3100, 36, 0.97), (6000, 20, 0.98), (7600, 16, 0.98)])
@pytest.mark.parametrize("select, c, drop", [("rsai", 2, "none"), ("rsai", 9, "fixed"), ("spai", 3, "none")])
def test_long_columns(n, dense, fill, select, c, drop):
    A = long_columns(n, dense, fill, n)
    kw = dict(c=c, l_max={"rsai": 20 // c, "spai": 16}[select], eps=0.05, drop=drop, tol=1e-2, select=select)
    ref = oracle.build(A, **kw)
    h, _, res, rho, loops, flags, st = gpu_M(A, precision="fp64", **kw)
    assert st["p_max"] >= 32 and st["q_max"] >= 0.99 * n and st["cols_bin"][2] >= dense and st["n_failed"] == 0
    assert_fp64_parity(A, ref, res, rho, loops, flags, st, rtol=1e-9)
    h.free()
    h, _, res, rho, *_ = gpu_M(A, precision="fp32_refine", **kw)
    check_fp32_every_column(A, res, rho, ref)
    h.free()
