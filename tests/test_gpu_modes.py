"""Field combination and mode projection over mode counts around the kernels'
group of 8, for both record types, with 16-byte aligned tensors and with
tensors one element off (the kernels' scalar form), against torch in FP64.

Tolerance: each result is a sum of M (combination) or E (projection) products
in FP64, so at most (terms + 2) 2^-53 times the sum of their magnitudes, plus
half an ulp of the record type for the combination's store.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2007_14401_gb300 import gcb
    return gcb


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("modes", [1, 7, 8, 9, 64])
@pytest.mark.parametrize("off", [0, 1])
def test_combine_and_project(G, dtype, modes, off):
    import torch
    ny, nx = 5, 7
    Z = np.zeros((ny, nx))
    grid = G.Grid(dict(E=[Z] * 3, B=[Z] * 3, dB=[Z] * 6, dx=(1.0, 1.0)), dtype=dtype)
    n = grid.rec.numel()
    tdt = grid.rec.dtype
    gen = torch.Generator(device="cuda").manual_seed(modes)

    def tensor(shape, dt):
        k = int(np.prod(shape))
        return torch.empty(k + off, dtype=dt, device="cuda")[off:].view(shape).normal_(generator=gen)

    base, pat = tensor((n,), tdt), tensor((modes, n), tdt)
    pat[:, ::5] = 0.0
    pat[0, 3], pat[0, 4] = float("inf"), float("nan")
    amps = torch.randn(modes, generator=gen, dtype=torch.float64, device="cuda")
    G.grid_combine(grid, base, pat, amps)
    terms = amps[:, None] * pat.double()
    want = base.double() + terms.sum(0)
    mag = base.double().abs() + terms.abs().sum(0)
    ok = torch.isfinite(want)
    err = (grid.rec.double() - want).abs()
    half = want.abs() * (2.0 ** -24 if dtype == "f32" else 2.0 ** -53)
    assert bool((err[ok] <= ((modes + 2) * 2.0 ** -53 * mag + half)[ok]).all())
    assert int((~ok).sum()) == 2
    assert bool(torch.isinf(grid.rec[3])) and bool(torch.isnan(grid.rec[4]))
    pat[0, 3] = pat[0, 4] = 1.0
    grad = tensor((n,), torch.float64)
    got = G.grad_project(grid, grad, pat)
    terms = grad * pat.double()
    assert bool(((got - terms.sum(1)).abs() <= (n + 2) * 2.0 ** -53 * terms.abs().sum(1)).all())
