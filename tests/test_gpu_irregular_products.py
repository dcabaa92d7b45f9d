"""Products with rows of very different lengths: rows side by side, long rows apart and one row per
group give the same sums, for any length, number of rows and average."""
import numpy as np
import pytest

from paper_1503_04500_gb300 import inputs as gen
from test_gpu_solver_sizes import matvec, reference

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
rsai = pytest.importorskip("paper_1503_04500_gb300.rsai")

# around the rounds of 8 lanes, the limit of a short row and the entries in flight
LENGTHS = [0, 1, 7, 8, 9, 16, 17, 23, 24, 25, 31, 32, 33, 55, 56, 57, 64, 65, 257]


def rows_of(n, lengths):
    """(row_ptr, col_idx) with lengths[i % len] entries in row i, spread over the columns."""
    k = np.minimum(np.asarray(lengths)[np.arange(n) % len(lengths)], n)
    ptr = np.concatenate([[0], np.cumsum(k)]).astype(np.int64)
    row = np.repeat(np.arange(n), k)
    at = np.arange(ptr[-1]) - ptr[row]
    return ptr, ((row + at * np.maximum(n // np.maximum(k[row], 1), 1)) % n).astype(np.int32)


@pytest.mark.parametrize("lengths", [LENGTHS, LENGTHS + [3] * 12, [5] * 15 + [200], [25] * 9 + [2] * 8,
                                     [25, 3, 400, 24] * 3 + [80], [0] * 5 + [1]])
@pytest.mark.parametrize("n", [6, 7, 16, 17, 1000, 12288, 12289, 65536, 65537])
def test_every_length(n, lengths):
    """Whole numbers: every order of the additions gives the exact sum."""
    ptr, idx = rows_of(n, lengths)
    rng = np.random.default_rng(n)
    val = rng.integers(-8, 9, idx.size).astype(np.float64)
    x = rng.integers(-1000, 1001, n).astype(np.float64)
    want = np.bincount(np.repeat(np.arange(n), np.diff(ptr)), weights=val * x[idx], minlength=n)
    y = torch.full((n + 8,), 7.0, dtype=torch.float64, device="cuda")
    rsai.spmv(*(torch.as_tensor(t, device="cuda") for t in (ptr, idx, val, x)), y=y)
    np.testing.assert_array_equal(y.cpu().numpy(), np.concatenate([want, np.full(8, 7.0)]))


@pytest.mark.parametrize("long_A", [False, True])
@pytest.mark.parametrize("n", [100, 3000, 20011])
def test_solve_with_long_rows_of_m(n, long_A):
    """M of 40 entries per row and a few of hundreds: its products take more blocks than the vectors."""
    A = gen.powerlaw(n, seed=n, dmin=40 if long_A else 3, dmax=min(n - 1, 200))
    rng = np.random.default_rng(n)
    ptr, idx = rows_of(n, [40] * 30 + [600])
    row = np.repeat(np.arange(n), np.diff(ptr))
    diag = np.zeros(n)
    entry = np.repeat(np.arange(n), np.diff(A.row_ptr)) == A.col_idx
    diag[A.col_idx[entry]] = A.val[entry]
    val = np.where(idx == row, 1.0, rng.standard_normal(idx.size) * 1e-3) / diag[row]
    M = gen.SparseMatrix(n, ptr, idx, val, None, None, None, None)
    apply_M = lambda z: matvec(M, z)  # noqa: E731
    b = rng.standard_normal(n)
    x = torch.empty(n, dtype=torch.float64, device="cuda")
    iters, relres, status = rsai.bicgstab_noalloc(rsai.DeviceMatrix.from_host(A),
                                                  tuple(torch.as_tensor(t, device="cuda") for t in (ptr, idx, val)),
                                                  torch.as_tensor(b, device="cuda"), x, rtol=1e-14, maxit=3)
    # the bar of test_gpu_solver_sizes: rounding times the iteration's own sensitivity
    ref, _ = reference(A, apply_M, b, 1e-14, 3)
    moved, _ = reference(A, apply_M, b * (1 + 2.0**-52), 1e-14, 3)
    assert iters == 3 and status == 11
    x = x.cpu().numpy()
    assert np.abs(x - ref).max() <= 1e-10 * np.abs(ref).max() + 30 * np.abs(moved - ref).max()
    np.testing.assert_allclose(relres, np.linalg.norm(b - matvec(A, x)) / np.linalg.norm(b), rtol=1e-9, atol=1e-13)
