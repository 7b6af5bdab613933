"""The FP64 reciprocals, roots and penalty norm of f64math.cuh, compiled into a
small library of their own, against extended precision.

Bounds, with the seeds' documented errors (reciprocal 1 ulp, inverse square
root 2^-22.9): the third-order step leaves less than 1e-18 and the last
multiply-add rounds once, so reciprocals and inverse roots are within one unit
in the last place; the square root multiplies a rounded inverse root by x and
rounds again, two units.  Outside [2^-959, 2^960) and for zero, subnormal,
infinite, NaN and negative arguments they are CUDA's own operations, each
rounded correctly.

The norm is q + 2 p w of the trigonometric solution: 1e-12 relative away from
the double root (r is known to some 1e-15, and dw/dr is at most 17 where the
Newton steps are taken), and where the two largest eigenvalues meet the square
root of that, 1e-7.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2508_17917_gb300", "csrc")
SOURCE = r"""
#include "f64math.cuh"
__global__ void unary(int which, const double *x, double *y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = which == 0 ? dg::rcp64(x[i]) : which == 1 ? dg::rsqrt64(x[i]) : dg::sqrt64(x[i]);
}
__global__ void norm(const double *s, double gPr, double *y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    dg::Phys<double> ph{};
    ph.mu = 1.0;
    ph.gPr = gPr;
    const double *q = s + 5 * i;
    y[i] = dg::penalty_norm64(1.0, q[0], q[1], q[2], q[3], q[4], ph);
}
extern "C" int run_unary(int which, const double *x, double *y, int n)
{
    unary<<<(n + 127) / 128, 128>>>(which, x, y, n);
    return cudaDeviceSynchronize();
}
extern "C" int run_norm(const double *s, double gPr, double *y, int n)
{
    norm<<<(n + 127) / 128, 128>>>(s, gPr, y, n);
    return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_17917_gb300 import build
    d = tmp_path_factory.mktemp("f64")
    (d / "f64.cu").write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", CSRC, "-shared", "-cudart", "shared", "-o",
                    str(d / "f64.so"), str(d / "f64.cu")], check=True)
    return C.CDLL(str(d / "f64.so"))


def unary(lib, which, x):
    import torch
    a = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    y = torch.empty_like(a)
    assert lib.run_unary(which, C.c_void_p(a.data_ptr()), C.c_void_p(y.data_ptr()), a.numel()) == 0
    return y.cpu().numpy()


def ulps(got, exact):
    return np.abs((np.longdouble(got) - exact) / np.spacing(np.abs(exact.astype(np.float64)))).max()


def arguments():
    rng = np.random.default_rng(5)
    m = np.concatenate([rng.uniform(1, 2, 200_000), 1 + 2.0 ** -np.arange(1, 53), 2 - 2.0 ** -np.arange(1, 53)])
    return np.concatenate([m, m[:20_000] * 2.0 ** rng.integers(-1000, 1000, 20_000),
                           *(np.array([1.0, 1.5, 1.9999]) * 2.0 ** e for e in (-1021, -960, -959, -958, 957, 958, 959,
                                                                               1000, 1022))])


def test_reciprocal(lib):
    x = arguments()
    x = np.concatenate([x, -x])
    assert ulps(unary(lib, 0, x), 1 / np.longdouble(x)) <= 1.0


def plain(x):
    return (np.abs(x) >= 2.0 ** -959) & (np.abs(x) < 2.0 ** 960)


def test_roots(lib):
    x = arguments()
    out = x[~plain(x)]
    assert np.array_equal(unary(lib, 1, out), 1 / np.sqrt(out)) and np.array_equal(unary(lib, 2, out), np.sqrt(out))
    x = x[plain(x)]
    root = np.sqrt(np.longdouble(x))
    assert ulps(unary(lib, 1, x), 1 / root) <= 1.0
    assert ulps(unary(lib, 2, x), root) <= 2.0


def test_special_arguments(lib):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.0 ** -1030, -1.0, -2.0 ** -1000])
    with np.errstate(all="ignore"):
        for which, ref in ((0, 1 / x), (1, 1 / np.sqrt(x)), (2, np.sqrt(x))):
            assert np.array_equal(unary(lib, which, x), ref, equal_nan=True), which


def exact_norm(v1, v2, e, n1, n2, g):
    vn, vt, vsq = v1 * n1 + v2 * n2, v2 * n1 - v1 * n2, v1 * v1 + v2 * v2
    a41, c42, c43 = -vn * vn / 3 - vsq - g * (e - vsq), (4 / 3 - g) * vn, (1 - g) * vt
    S = np.empty(vn.shape + (3, 3))
    S[..., 0, 0], S[..., 1, 1] = 16 / 9 * (vn * vn + 1), vt * vt + 1
    S[..., 2, 2] = a41 ** 2 + c42 ** 2 + c43 ** 2 + g * g
    S[..., 0, 1] = S[..., 1, 0] = 4 / 3 * vn * vt
    S[..., 0, 2] = S[..., 2, 0] = 4 / 3 * (c42 - vn * a41)
    S[..., 1, 2] = S[..., 2, 1] = c43 - vt * a41
    lam = np.linalg.eigvalsh(S)
    return np.sqrt(lam[..., 2]), 1.0 - lam[..., 1] / lam[..., 2]      # and the gap to the next one


@pytest.mark.parametrize("g", [0.7, 1.0, 1.4 / 0.72])
def test_penalty_norm(lib, g):
    import torch
    rng = np.random.default_rng(6)
    n = 200_000
    speed, th, an = np.exp(rng.uniform(-12, 2, n)), rng.uniform(0, 2 * np.pi, n), rng.uniform(0, 2 * np.pi, n)
    e = np.exp(rng.uniform(-3, 4, n)) + 0.5 * speed ** 2
    if g < 4 / 3:                                     # around the double root at rest
        k = n // 2
        e[:k] = np.sqrt((4 / 3 / g) ** 2 - 1) * (1 + rng.normal(size=k) * np.exp(rng.uniform(-25, -2, k)))
        speed[:k] = np.exp(rng.uniform(-12, -4, k))
    s = np.stack([speed * np.cos(th), speed * np.sin(th), e, np.cos(an), np.sin(an)], 1)
    ref, gap = exact_norm(*s.T, g)
    a = torch.from_numpy(np.ascontiguousarray(s)).cuda()
    y = torch.empty(n, dtype=torch.float64, device="cuda")
    assert lib.run_norm(C.c_void_p(a.data_ptr()), C.c_double(g), C.c_void_p(y.data_ptr()), n) == 0
    err = np.abs(y.cpu().numpy() / ref - 1.0)
    assert err.max() <= 1e-7
    assert err[gap > 0.05].max() <= 1e-12
