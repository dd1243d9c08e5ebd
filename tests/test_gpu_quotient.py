"""plain::quotient (a division by a number whose reciprocal is at hand, in the FP64 kernels) against the
device's own IEEE division, bit for bit, the sign of a zero included: random operands, mantissas at both
ends of a binade, dividends and divisors around the exponents beyond which the division itself runs, zeros,
subnormals, infinities and NaN."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2504_15018_gb300 import builder

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "plb_plain.cuh"
__global__ void k(const double *a, const double *b, long long n, double *q, double *d) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    q[i] = plb::plain::quotient(a[i], b[i], plb::plain::reciprocal(b[i]));
    d[i] = a[i] / b[i];
}
extern "C" int run(const double *a, const double *b, long long n, double *q, double *d) {
    double *buf;
    if (cudaMalloc(&buf, 4 * n * sizeof(double)) != cudaSuccess) return 1;
    cudaMemcpy(buf, a, n * sizeof(double), cudaMemcpyHostToDevice);
    cudaMemcpy(buf + n, b, n * sizeof(double), cudaMemcpyHostToDevice);
    k<<<(unsigned)((n + 255) / 256), 256>>>(buf, buf + n, n, buf + 2 * n, buf + 3 * n);
    cudaMemcpy(q, buf + 2 * n, n * sizeof(double), cudaMemcpyDeviceToHost);
    cudaMemcpy(d, buf + 3 * n, n * sizeof(double), cudaMemcpyDeviceToHost);
    cudaFree(buf);
    return cudaGetLastError() != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("quotient")
    src, so = d / "q.cu", d / "q.so"
    src.write_text(SOURCE)
    subprocess.run([builder._nvcc(), *builder.ARCH, *builder.COMMON, "-fmad=false", "-shared", "-o", str(so), str(src)],
                   check=True)
    fn = ctypes.CDLL(str(so)).run
    dp = ctypes.POINTER(ctypes.c_double)
    fn.argtypes = [dp, dp, ctypes.c_longlong, dp, dp]

    def divide(a, b):
        a, b = (np.ascontiguousarray(v, dtype=np.float64) for v in (a, b))
        q, w = np.empty_like(a), np.empty_like(a)
        assert fn(*(v.ctypes.data_as(dp) for v in (a, b)), a.size, *(v.ctypes.data_as(dp) for v in (q, w))) == 0
        return q, w
    return divide


def _assert_same(q, w):
    same = (q.view(np.uint64) == w.view(np.uint64)) | (np.isnan(q) & np.isnan(w))
    assert same.all(), (np.flatnonzero(~same)[:5], q[~same][:5], w[~same][:5])


def _mantissas(rng, n):
    """Random mantissas in [1, 2), a third of them within 64 units of either end."""
    m = rng.randint(0, 1 << 52, n, dtype=np.int64)
    k = n // 3
    m[:k // 2] = rng.randint(0, 64, k // 2)
    m[k // 2:k] = (1 << 52) - 1 - rng.randint(0, 64, k - k // 2)
    return rng.permutation(1.0 + m * 2.0 ** -52)


@pytest.mark.parametrize("a_exp,b_exp", [(40, 4), (900, 3), (1022, 110), (3, 101)])
def test_random_operands(run, a_exp, b_exp):
    rng = np.random.RandomState(a_exp)
    n = 1 << 23
    sign = lambda: rng.choice([-1.0, 1.0], n)
    a = sign() * np.ldexp(_mantissas(rng, n), rng.randint(-a_exp, a_exp + 1, n))
    b = sign() * np.ldexp(_mantissas(rng, n), rng.randint(-b_exp, b_exp + 1, n))
    _assert_same(*run(a, b))


def test_divisors_in_use(run):
    """3, relaxation times, G, density spans, against quotients one unit beside a midpoint and a double."""
    rng = np.random.RandomState(2)
    n = 1 << 22
    b = rng.choice(np.r_[3.0, -1.0, -0.37, 0.56, 0.62873, 0.8, 1.0, 1.1, 6.98, 1.1495, rng.uniform(0.5, 2, 32)], n)
    q = np.ldexp(_mantissas(rng, n), rng.randint(-20, 20, n))
    a = q * b
    a = np.where(rng.rand(n) < 0.5, a, np.nextafter(a, rng.choice([-np.inf, np.inf], n)))
    _assert_same(*run(a, b))


def test_limits(run):
    e = np.r_[-1074, -1060:-1015, -905:-890, -5:5, 890:905, 1015:1024]
    a = np.unique(np.r_[np.ldexp(1.0, e), np.ldexp(1.9999999999999998, np.clip(e, -1074, 1023)), np.ldexp(1.25, e)])
    f = np.r_[-1074, -1022, -105:-95, -2:3, 95:105, 1022, 1023]
    b = np.unique(np.r_[np.ldexp(1.0, f), np.ldexp(1.9999999999999998, f), np.ldexp(1.3, f), 3.0])
    a, b = (np.r_[v, -v, 0.0, -0.0, np.inf, -np.inf, np.nan] for v in (a, b))
    A, B = np.meshgrid(a, b)
    _assert_same(*run(A.ravel(), B.ravel()))
