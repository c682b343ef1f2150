"""An axis longer than the 2^22 cells that the FP32 gather's short floor covers,
with fields of period 16 along it, so that every step has its twin on an axis of
16 cells.

Offsets of 2^22 cells and more (a half-step point that far from its particle,
in half cells, which a float resolves there): bit for bit as the twin, whose
offset is the same modulo 16.  Particles in the last cells, the last one's upper
neighbour among them: their base cell, and with it the rounding of an offset,
depends on where a float of 2^22 puts them, so within rounding (1e-5, about 100
roundings), but for one in a thousand whose point crosses a face, where the
gradient of the shape functions jumps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NY = 4
LONG = (1 << 22) + 16


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2007_14401_gb300 import gcb
    return gcb


@pytest.fixture(scope="module")
def grids(G):
    out = {}
    for nx in (16, LONG):
        X = 2 * np.pi * np.arange(nx)[None, :] / 16 * np.ones((NY, 1))
        Y = np.pi * np.arange(NY)[:, None] / 2 * np.ones((1, nx))
        # the same bits in every period
        f = [np.tile(c[:, :16], (1, nx // 16)) for c in
             (0.1 * np.sin(X), 0.1 * np.cos(Y), 0.1 * np.cos(X + Y),
              0.3 * np.sin(Y), 0.3 * np.cos(X), 1.0 + 0.2 * np.sin(X - Y))]
        out[nx] = G.Grid(dict(E=f[:3], B=f[3:], dB=None, dx=(1.0, 1.0)), dtype="f32")
    return out


def step(G, grid, x, y, u, dxp):
    st = dict(x=np.stack([x, y]), u=u, dxp=dxp, flags=np.zeros(x.size, np.uint8))
    ds = G.State.from_numpy(st, precision="mixed", pos_mode="pair")
    p = dict(qm=(100.0,), dt=0.4, dl=1.0, f_rho=0.4, grad_mode=0, gca_fixed_iters=5)
    s = G.push(ds, grid, G.make_params(p), 1)
    assert s["n_gca"] == x.size
    return ds.u.cpu().numpy(), ds.dxp.cpu().numpy()


@pytest.mark.parametrize("sign", [1, -1])
def test_offsets_past_the_short_floor(G, grids, sign):
    n = 4000
    rng = np.random.default_rng(8)
    u = rng.normal(size=(3, n))
    near = rng.integers(0, 24, n) / 2.0                     # 0 .. 11.5 cells
    y = rng.integers(0, NY * 1024, n) / 1024.0
    # base cells from which the point stays inside the long axis, and any
    x = np.where(np.arange(n) % 2, rng.integers(0, 4, n), rng.integers(0, 16, n)).astype(float)
    if sign < 0:
        x = LONG - 16.0 + 15.0 - x
    dy = 0.4 * u[1] / np.sqrt(1 + (u ** 2).sum(0))
    a = step(G, grids[LONG], x, y, u, np.stack([-2.0 * sign * ((1 << 22) + near), dy]))
    b = step(G, grids[16], x % 16, y, u, np.stack([-2.0 * sign * near, dy]))
    for p, q in zip(a, b):
        np.testing.assert_array_equal(p, q)


def test_last_cells(G, grids):
    n = 20000
    rng = np.random.default_rng(9)
    u = rng.normal(size=(3, n))
    xs = rng.integers(0, 16 * 1024, n) / 1024.0
    xs[:5000] = 15.0 + rng.integers(0, 1024, 5000) / 1024.0  # the last cell
    y = rng.integers(0, NY * 1024, n) / 1024.0
    dxp = 0.4 * u[:2] / np.sqrt(1 + (u ** 2).sum(0))
    a = step(G, grids[LONG], xs + (LONG - 16.0), y, u, dxp)
    b = step(G, grids[16], xs, y, u, dxp)
    bad = (np.abs(a[0] - b[0]) > 1e-5 * (1.0 + np.linalg.norm(b[0], axis=0))).any(0)
    bad |= (np.abs(a[1] - b[1]) > 1e-5).any(0)
    assert bad.mean() < 1e-3
