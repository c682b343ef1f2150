"""The FP64 building blocks of csrc/real64.cuh against extended precision.

Reciprocal, reciprocal root and root over the exponent range (tolerances from
the iteration: a third-order step from a 20-bit start leaves 2^-58, so the
last rounding decides: 1 ulp, the root 2), their limits at 0, infinity and
NaN, and the floor with its clamped integer, exact at and around integers.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2007_14401_gb300", "csrc")
SRC = r"""
#include "real64.cuh"
__global__ void k(long n, const double *x, double *o, int *ki, int lim)
{
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        o[i] = gcb::rcp64(x[i]);
        o[n + i] = gcb::rsqrt64(x[i]);
        o[2 * n + i] = gcb::sqrt64(x[i]);
        o[3 * n + i] = gcb::floor64(x[i], lim, ki[i]);
    }
}
extern "C" int run(long n, const double *x, double *o, int *ki, int lim)
{
    k<<<64, 256>>>(n, x, o, ki, lim);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("real64")
    (d / "t.cu").write_text(SRC)
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "-I" + CSRC, "-shared", "-Xcompiler", "-fPIC", str(d / "t.cu"), "-o",
                    str(d / "t.so")], check=True)
    lib = ctypes.CDLL(str(d / "t.so"))

    def f(x, lim=1000):
        t = torch.tensor(x, dtype=torch.float64, device="cuda")
        o = torch.zeros((4, t.numel()), dtype=torch.float64, device="cuda")
        k = torch.zeros(t.numel(), dtype=torch.int32, device="cuda")
        p = ctypes.c_void_p
        assert lib.run(ctypes.c_long(t.numel()), p(t.data_ptr()), p(o.data_ptr()),
                       p(k.data_ptr()), lim) == 0
        return o.cpu().numpy(), k.cpu().numpy()
    return f


@pytest.mark.parametrize("lo,hi", [(-1e-9, 1e-9), (-1.0, 1.0), (-60.0, 60.0), (-1000.0, 1000.0)])
def test_reciprocals_and_roots(run, lo, hi):
    rng = np.random.default_rng(3)
    x = 2.0 ** rng.uniform(lo, hi, 200000) * rng.uniform(1.0, 2.0, 200000)
    x[:4] = [1.0, np.nextafter(1.0, 2.0), np.nextafter(1.0, 0.0), 4.0]
    (r, q, s, _), _ = run(x)
    X = x.astype(np.longdouble)
    for got, want, ulps in ((r, 1 / X, 1.0), (q, 1 / np.sqrt(X), 1.0), (s, np.sqrt(X), 2.0)):
        err = np.abs(got.astype(np.longdouble) - want) / np.spacing(want.astype(np.float64))
        assert float(err.max()) <= ulps
    (rn, _, _, _), _ = run(-x)
    assert np.array_equal(rn, -r)


def test_limits(run):
    (r, q, s, _), _ = run([0.0, np.inf, np.nan, -1.0, 1e-320, -np.inf])
    assert r[0] == np.inf and r[1] == 0.0 and np.isnan(r[2]) and r[5] == 0.0
    assert q[0] == np.inf and q[1] == 0.0 and np.isnan(q[2]) and np.isnan(q[3]) and q[4] == np.inf
    assert s[0] == 0.0 and s[1] == np.inf and np.isnan(s[2]) and np.isnan(s[3]) and np.isnan(s[5])


@pytest.mark.parametrize("lim", [7, 1000, 2 ** 31 - 1])
def test_floor_and_clamp(run, lim):
    rng = np.random.default_rng(4)
    k = np.concatenate([np.arange(-12.0, 13.0), rng.integers(-2 ** 40, 2 ** 40, 1000).astype(float)])
    x = np.concatenate([k, np.nextafter(k, np.inf), np.nextafter(k, -np.inf),
                        rng.uniform(-2000, 2000, 10000), [-0.0, 1e-300, -1e-300]])
    (_, _, _, f), i = run(x, lim)
    assert np.array_equal(f, np.floor(x))
    assert np.array_equal(i, np.clip(np.floor(x), -lim, lim).astype(np.int64))
    _, i = run([1e300, -1e300, np.inf, -np.inf, np.nan], lim)
    assert list(i[:4]) == [lim, -lim, lim, -lim] and abs(int(i[4])) <= lim
