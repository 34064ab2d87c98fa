"""The Boys function of the fp64 lane kernels beyond its table (T >= 64, upward
recursion F_{m+1} = (2m+1) F_m / 2T) against extended precision.

Bound: the rms error of every order may be no more than 1.2 times that of the
same recursion with 1/T by division in fp64 -- both make the same number of
roundings a step, the rms of 4096 of them is known to 2 %, and the reciprocal
may carry one rounding more (sqrt(4/3) of it at most)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

M = 9
SRC = r"""
#include "eri_herm.cuh"
__global__ void k(int n, const double *T, double *F)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double f[%(M)d + 1];
    tg::boys_lane<%(M)d>(T[i], f, nullptr);  // T >= 64: the table is not read
    for (int m = 0; m <= %(M)d; ++m) F[m * n + i] = f[m];
}
extern "C" int run(int n, const double *T, double *F)
{
    k<<<(n + 127) / 128, 128>>>(n, T, F);
    return (int)cudaDeviceSynchronize();
}
""" % {"M": M}


@pytest.fixture(scope="module")
def boys(tmp_path_factory):
    torch = pytest.importorskip("torch")
    from paper_2407_16586_gb300 import build as b
    d = tmp_path_factory.mktemp("boys")
    src, so = os.path.join(d, "far.cu"), os.path.join(d, "far.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([b._nvcc()] + b.ARCH + b.FLAGS + ["-shared", src, "-o", so], check=True, capture_output=True)
    fn = ctypes.CDLL(so).run
    fn.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]

    def run(T):
        assert np.all(T >= 64.0)
        t = torch.from_numpy(T).cuda()
        F = torch.zeros((M + 1, len(T)), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert fn(len(T), t.data_ptr(), F.data_ptr()) == 0
        return F.cpu().numpy()
    return run


def _upward(T, f0):
    F = [f0]
    e = np.exp(-T)
    for m in range(M):
        F.append(((2 * m + 1) * F[m] - e) / (2 * T))
    return np.array(F)


@pytest.mark.parametrize("lo,hi", [(64.0, 128.0), (128.0, 1e3), (1e3, 1e8)])
def test_far_orders_are_as_accurate_as_by_division(boys, lo, hi):
    rng = np.random.default_rng(3)
    T = np.exp(rng.uniform(np.log(lo), np.log(hi), 4096)).clip(lo, hi)
    T[0] = lo
    X = T.astype(np.longdouble)
    pi = np.longdouble("3.14159265358979323846264338327950288")
    ref = _upward(X, np.sqrt(pi / X) / 2)
    h = 0.5 * (1.0 / T)
    plain = [0.88622692545275801365 * np.sqrt(1.0 / T)]
    for m in range(M):
        plain.append(((2 * m + 1) * plain[m] - np.exp(-T)) * h)

    def rms(F):
        return np.sqrt(np.mean(((F - ref) / ref).astype(np.float64) ** 2, axis=1))
    got, old = rms(boys(T)), rms(np.array(plain))
    # order 0 differs by 1/sqrt(T) itself: rsqrt to one ulp against sqrt(1/T)
    assert np.all(got <= 1.2 * old + 1e-17), (got, old)


def test_far_orders_at_infinity(boys):
    F = boys(np.array([64.0, 1e200, np.inf]))
    assert np.all(np.isfinite(F)) and np.all(F[:, 2] == 0.0)
