"""Cell and fraction of an FP64 coordinate (csrc/real64.cuh: split64) against
exact rational arithmetic: the integer is the floor of the unrounded product,
the fraction is its remainder rounded once (half an ulp of 1 at most), at and
around integers, with the integer's clamp, infinities and NaN."""
import ctypes
import subprocess
from fractions import Fraction
from math import floor
from pathlib import Path

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = Path(__file__).resolve().parent.parent / "paper_2007_14401_gb300" / "csrc"
SRC = r"""
#include "real64.cuh"
__global__ void k(int n, const double *l, double i, double *t, int *ki, int lim)
{
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
        t[j] = gcb::split64(l[j], i, lim, ki[j]);
}
extern "C" int run(int n, const double *l, double i, double *t, int *ki, int lim)
{
    k<<<8, 256>>>(n, l, i, t, ki, lim);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("split64")
    (d / "t.cu").write_text(SRC)
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "-I" + str(CSRC), "-shared", "-Xcompiler", "-fPIC", str(d / "t.cu"), "-o",
                    str(d / "t.so")], check=True)
    lib = ctypes.CDLL(str(d / "t.so"))

    def f(l, i, lim):
        x = torch.tensor(l, dtype=torch.float64, device="cuda")
        t = torch.zeros_like(x)
        k = torch.zeros(x.numel(), dtype=torch.int32, device="cuda")
        p = ctypes.c_void_p
        assert lib.run(x.numel(), p(x.data_ptr()), ctypes.c_double(i), p(t.data_ptr()),
                       p(k.data_ptr()), lim) == 0
        return t.cpu().numpy(), k.cpu().numpy()
    return f


@pytest.mark.parametrize("inv_dx", [1.0, 1.0 / 0.1, 512.0, 3.0 / 7.0, 1e-3])
@pytest.mark.parametrize("n", [2, 1000])
def test_floor_and_fraction(run, inv_dx, n):
    rng = np.random.default_rng(6)
    e = np.arange(-6.0, 7.0) / inv_dx
    l = np.concatenate([e, np.nextafter(e, np.inf), np.nextafter(e, -np.inf),
                        rng.uniform(-5.0, 5.0, 1500) / inv_dx, [-0.0, 1e-300, -1e-300, -1e-18]])
    t, k = run(l, inv_dx, n)
    for a, tt, kk in zip(l, t, k):
        s = Fraction(float(a)) * Fraction(inv_dx)
        assert kk == max(-n, min(n, floor(s)))
        assert 0.0 <= tt <= 1.0 and abs(Fraction(float(tt)) - (s - floor(s))) <= Fraction(1, 2 ** 54)
    _, k = run([1e300, -1e300, np.inf, -np.inf, np.nan], inv_dx, n)
    assert list(k[:4]) == [n, -n, n, -n] and abs(int(k[4])) <= n
