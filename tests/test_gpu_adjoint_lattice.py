"""Gather points on cell faces of a grid whose spacing is no power of two: the
offset times 1/dx rounds to an integer there, or does not, so that a cell and a
fraction taken from two roundings of it belong to different cells.  The two
constructions of the transposed FP64 step (written-out reverse sweep, dual
numbers) must see the same fields: equal to FP64 rounding, as on particles
placed at random."""
from fractions import Fraction
from math import floor

import numpy as np
import pytest

from paper_2007_14401_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2007_14401_gb300 import gcb
    return gcb


@pytest.mark.parametrize("dx", [0.1, 0.7])
def test_reverse_and_tangent_agree_on_faces(G, dx):
    import torch
    nx, ny = 16, 8
    X, Y = np.meshgrid(2 * np.pi * np.arange(nx) / nx, 2 * np.pi * np.arange(ny) / ny)
    B = [0.3 * np.sin(Y), 0.2 * np.cos(X), 1.0 + 0.3 * np.sin(X + Y)]
    fields = dict(E=[0.1 * np.sin(X), 0.1 * np.cos(Y), 0.05 * np.cos(X - Y)], B=B,
                  dB=inputs.central_gradients(B, (dx, dx)), dx=(dx, dx))
    # on nodes 0, 1, 2, 4 (offset from the base cell exactly 0), the half-step
    # point k cells back or on along each axis
    ks = np.arange(-7, 8)
    i, j, kx, ky = (v.ravel() for v in np.meshgrid([0, 1, 2, 4], [0, 2], ks, ks))
    n = i.size
    rng = np.random.default_rng(2)
    off = np.stack([kx * dx, ky * dx])
    two = [sum(floor(float(v) * (1.0 / dx)) != floor(Fraction(float(v)) * Fraction(1.0 / dx))
               for v in o) for o in off]
    assert min(two) > n // 50                      # cells the two roundings tell apart
    st = dict(x=np.stack([i * dx, j * dx]), u=rng.normal(size=(3, n)), dxp=-2.0 * off,
              flags=np.zeros(n, np.uint8))
    grid = G.Grid(fields, dtype="f64")
    gp = G.make_params(dict(qm=(1e4,), dt=0.3 * dx, dl=dx), grad_mode=1, gca_fixed_iters=4)
    lam0 = torch.randn((7, n), dtype=torch.float64, device="cuda",
                       generator=torch.Generator(device="cuda").manual_seed(1))
    ds = G.State.from_numpy(st, precision="fp64", pos_mode="f64")
    assert G.push(ds.clone(), grid, gp, 1)["n_gca"] == n
    out = {}
    for method in ("reverse", "tangent"):
        lam = lam0.clone()
        grad = G.adjoint(ds, grid, gp, 1, lam, 1, method=method)
        out[method] = lam.cpu().numpy(), grad.cpu().numpy()
    for a, b in zip(out["reverse"], out["tangent"]):
        np.testing.assert_allclose(a, b, rtol=0, atol=1e-11 * np.abs(a).max())
