"""The result pool of a first build: columns that find it full run again, M's arrays hold whatever
the pool holds, and a later rebuild with other values has the same room."""
import numpy as np
import pytest

import oracle
from paper_1503_04500_gb300 import inputs as gen
from parity_check import check_fp32_every_column
from test_gpu_failures import RSAI_ERR_OOM, FailingAllocator
from test_gpu_parity import assert_fp64_parity, gpu_M

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
rsai = pytest.importorskip("paper_1503_04500_gb300.rsai")


def arrow(m, seed):
    """Diagonal, a dense first row and a third of the first subdiagonal: |J| = m after one loop."""
    rng = np.random.default_rng(seed)
    i, s = np.arange(m), np.arange(1, m, 3)
    return gen.from_coo(m, np.concatenate([i, 0 * i[1:], s]), np.concatenate([i, i[1:], s - 1]),
                        np.concatenate([2 + rng.random(m), rng.standard_normal(m - 1), rng.standard_normal(s.size)]))


def block_diagonal(blocks):
    rows, cols, vals, n = [], [], [], 0
    for m in blocks:
        rows.append(np.repeat(np.arange(m.n), np.diff(m.row_ptr)) + n)
        cols.append(m.col_idx.astype(np.int64) + n)
        vals.append(m.val)
        n += m.n
    return gen.from_coo(n, *(np.concatenate(x) for x in (rows, cols, vals)))


KW = dict(c=8, l_max=8, eps=1e-3, drop="none")


def first_estimate(A):
    """Entries of the pool that a build starts with."""
    return min(A.n * max(32, 10 * (A.nnz // A.n) + 16), A.n**2)


def full_before_the_global_bin():
    """600 columns of 120 entries each in the shared-memory bins fill the pool (36 entries per
    column); nearly all of the other 500 reach the global bin, with 140 entries each."""
    return block_diagonal([arrow(120, 10 + i) for i in range(5)] + [gen.powerlaw(500, seed=77, dmin=2, dmax=4,
                                                                              dominance=0.3)])


def long_columns():
    """All columns reach the global bin, with 450 entries each: more than it makes room for."""
    return block_diagonal([arrow(450, 3), arrow(450, 4)])


def capacity(fa, nnz):
    """The entries that the pool (4 + 8 bytes per entry) and M's arrays (three of 4 bytes,
    five of 8) hold; they hold the same number."""
    sizes = list(fa.live.values())
    found = {b // 8 for b in sizes if b >= 8 * nnz and sizes.count(b) >= 6 and sizes.count(b // 2) >= 4}
    assert len(found) == 1, sorted(sizes)
    return found.pop()


@pytest.mark.parametrize("precision", ["fp64", "fp32_refine"])
@pytest.mark.parametrize("problem", [full_before_the_global_bin, long_columns])
def test_columns_that_find_the_pool_full_run_again(problem, precision):
    """A rerun happened (its list of columns was allocated); M is the oracle's; a rebuild
    with other values is the same as a first build with them."""
    A = problem()
    ref = oracle.build(A, **KW)
    assert ref.nnz > first_estimate(A)
    with FailingAllocator() as fa:
        h, dA, res, rho, loops, flags, st = gpu_M(A, precision=precision, **KW)
        assert 4 * A.n in fa.live.values()
        assert capacity(fa, st["nnz_M"]) >= st["nnz_M"]
        assert st["n_failed"] == 0
        if precision == "fp64":
            assert_fp64_parity(A, ref, res, rho, loops, flags, st, rtol=1e-9)
        else:
            # condition numbers of the LS problems up to 131, |J| up to 450: the residual that an FP32
            # factorization corrected once leaves is (131 sqrt(450) 2^-24)^2 = 3e-8
            check_fp32_every_column(A, res, rho, ref, rtol_rho=1e-3, rtol_val=1e-3, atol_rho=1e-7)
        val = dA.val * torch.linspace(0.9, 1.1, A.nnz, dtype=torch.float64, device="cuda")
        h.set_values(val)
        h.rebuild()
        got = [t.cpu().numpy() for t in h.M()]
        h.free()
    fresh = rsai.build(rsai.DeviceMatrix.from_host(A.with_values(val.cpu().numpy())), precision=precision, **KW)
    for a, b in zip(got, fresh.M()):
        np.testing.assert_array_equal(a, b.cpu().numpy())
    fresh.free()


class Requests(dict):
    """What is outstanding, and the size of every request so far."""

    def __init__(self):
        super().__init__()
        self.sizes = []

    def __setitem__(self, ptr, nbytes):
        self.sizes.append(nbytes)
        super().__setitem__(ptr, nbytes)


@pytest.mark.parametrize("precision", ["fp64", "fp32_refine"])
@pytest.mark.parametrize("problem, kw, reruns", [
    (lambda: gen.powerlaw(500, seed=3), dict(c=5, l_max=8, eps=0.4, drop="fixed"), False),  # fits the estimate
    (lambda: gen.powerlaw(600, seed=5, dmax=40), dict(c=5, l_max=6, eps=0.05, drop="none"), False),  # does not
    (long_columns, KW, True)])
def test_room_for_the_global_bin_is_bounded_and_given_back(precision, problem, kw, reruns):
    """Room for the global bin's columns is made (at most four times the estimate) and given
    back: the handle keeps the estimate, or twice the entries that did not fit it."""
    A = problem()
    cap = first_estimate(A)
    with FailingAllocator() as fa:
        fa.live = Requests()
        h = rsai.build(rsai.DeviceMatrix.from_host(A), precision=precision, **kw)
        st = h.stats()
        nnz, room = st["nnz_M"], st["cols_bin"][2] * 256
        kept = capacity(fa, nnz)
        if reruns:
            assert 8 * 4 * cap in fa.live.sizes and kept >= min(2 * nnz + 1024, A.n**2)
        else:
            assert any(8 * max(cap, room) < b <= 8 * 4 * cap for b in fa.live.sizes)
            assert kept == (cap if nnz <= cap else min(2 * nnz + 1024, max(A.n**2, nnz + 1024)))
        h.free()


@pytest.mark.parametrize("problem", [full_before_the_global_bin, long_columns])
def test_every_failed_allocation_of_a_rerun_is_oom_and_leaks_nothing(problem):
    dA = rsai.DeviceMatrix.from_host(problem())
    with FailingAllocator() as ok:
        rsai.build(dA, precision="fp64", **KW).free()
    torch.cuda.synchronize()
    assert ok.live == {}
    for n_fail in range(1, ok.calls + 1):
        with FailingAllocator(n_fail) as fa:
            with pytest.raises(rsai.RSAIError) as e:
                rsai.build(dA, precision="fp64", **KW)
            assert e.value.status == RSAI_ERR_OOM, n_fail
            torch.cuda.synchronize()
            assert fa.live == {}, (n_fail, len(fa.live))
