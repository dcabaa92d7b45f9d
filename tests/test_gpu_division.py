"""The FP64 quotients of the triangular solves and reflectors against CUDA's division, bit for bit."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1503_04500_gb300 import build_ext

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

KERNEL = """
#include "team_qr.cuh"
// out: a / d by Divisor and by the compiler's division, 2 / d by two_over_of and by the division
__global__ void k_quotients(const double *a, const double *d, double *out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = rsai::Divisor<double>(d[i]).into(a[i]);
    out[n + i] = a[i] / d[i];
    out[2 * (size_t)n + i] = rsai::two_over_of(d[i]);
    out[3 * (size_t)n + i] = 2.0 / d[i];
}
extern "C" int quotients(const double *a, const double *d, double *out, int n) {
    k_quotients<<<(n + 255) / 256, 256>>>(a, d, out, n);
    return cudaDeviceSynchronize() != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def quotients(tmp_path_factory):
    torch.zeros(1, device="cuda")
    d = tmp_path_factory.mktemp("division")
    (d / "q.cu").write_text(KERNEL)
    lib = str(d / "libq.so")
    subprocess.run([build_ext.nvcc(), *build_ext.ARCH, *build_ext.FLAGS, "-shared", "-I", build_ext.SRC, str(d / "q.cu"),
                    "-o", lib], check=True, capture_output=True)
    f = ctypes.CDLL(lib).quotients
    f.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]

    def run(a, d):
        a, d = (torch.as_tensor(np.ascontiguousarray(x), device="cuda") for x in (a, d))
        out = torch.empty(4, a.numel(), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert f(a.data_ptr(), d.data_ptr(), out.data_ptr(), a.numel()) == 0
        return out.cpu().numpy()

    return run


def same(got, want, *at):
    """Equal bits, any NaN equal to any other."""
    bad = (got.view(np.int64) != want.view(np.int64)) & ~(np.isnan(got) & np.isnan(want))
    assert not bad.any(), [(float(x[bad][0]).hex() if np.isfinite(x[bad][0]) else x[bad][0]) for x in (got, want, *at)]


def check(quotients, a, d):
    q = quotients(a, d)
    same(q[0], q[1], a, d)
    pos = d >= 0  # two_over_of takes v^T v > 0
    same(q[2][pos], q[3][pos], d[pos])


def test_special_values(quotients):
    """Zeros of both signs, the ends of the range, of the subnormals and of the direct
    quotient's exponents (2^-500 and 2^500), infinities and NaN, each over each."""
    ends = [2.0**e for e in (-1074, -1073, -1023, -1022, -501, -500, -499, -1, 0, 1, 499, 500, 501, 1020, 1021, 1022, 1023)]
    v = [0.0, np.inf, np.nan, np.finfo(float).max, 1.0 / 3.0, 3.0]
    for x in ends:
        v += [x, np.nextafter(x, np.inf), np.nextafter(x, 0.0), 1.5 * x if x < 2.0**1023 else x]
    v = np.array(v)
    v = np.concatenate([v, -v])
    a, d = np.meshgrid(v, v)
    check(quotients, a.ravel(), d.ravel())


@pytest.mark.parametrize("near", ["any", "one", "two"])
def test_random_values(quotients, near):
    """Random mantissas (any, just above 1, just below 2) at exponents within and across the
    direct quotient's range."""
    rng = np.random.default_rng(3)
    n = 1 << 21

    def mantissa():
        if near == "any":
            return rng.integers(0, 1 << 52, n)
        m = rng.integers(0, 1 << 10, n)
        return m if near == "one" else (1 << 52) - 1 - m

    for span in (40, 520, 1020):
        exponent = lambda: rng.integers(1023 - span, 1024 + span, n)  # noqa: E731
        a, d = ((mantissa() | (exponent() << 52) | (rng.integers(0, 2, n) << 63)).view(np.float64) for _ in range(2))
        check(quotients, a, d)
