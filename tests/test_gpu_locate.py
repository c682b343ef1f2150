"""Where the FP32 gather finds its cell: points on cell faces, in the first
and last cells of the box (where the upper neighbour or the whole cell wraps)
and on an axis longer than the 2^22 nodes the short form of the floor covers.

Edges: one mixed-precision step against the FP64 oracle within the tolerances
of the mixed parity tests (the interpolant is continuous across faces, so a
point filed in either neighbour gives the same field; gradients of the shape
functions are not, so with those the points stay a little off the faces).
Long axis: fields constant along it and positions exact in one float (beyond
2^22 a float resolves half a cell, and a particle's base cell and the rounding
of its offset depend on where that puts it), so the step must equal, bit for
bit, the same particles' step on a short axis.
"""
import numpy as np
import pytest

from paper_2007_14401_gb300 import inputs
from tests.helpers import periodic_diff
from tests.test_gpu_parity import run_both

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2007_14401_gb300 import gcb
    return gcb


def edge_positions(n, dims, off, seed):
    """Every coordinate on a face of the first, second, last but one or last
    cell (+- off), or in the middle of one of them."""
    rng = np.random.default_rng(seed)
    x = np.empty((len(dims), n))
    for d, L in enumerate(dims):
        face = rng.choice([0.0, 1.0, L - 2.0, L - 1.0], n)
        x[d] = np.mod(face + rng.choice([off, -off, 0.5], n), L)
    return x


@pytest.mark.parametrize("kind", ["grid2d", "dw2d", "dw3d"])
def test_edges_against_oracle(G, kind):
    if kind == "dw3d":
        fields, st, p = inputs.current_sheet_3d(n=24, n_particles=4001, seed=3)
        dims, over = (24, 24, 24), dict(gca_fixed_iters=5)
    else:
        fields, st, p = inputs.reconnection_2d(nx=64, ny=32, n_particles=4001, seed=3)
        p = dict(p, qm=tuple(q * 1e-3 for q in p["qm"]))
        dims, over = (64, 32), dict(gca_fixed_iters=5, grad_mode=1 if kind == "grid2d" else 0)
    st["x"] = edge_positions(4001, dims, 0.0 if kind == "grid2d" else 0.03125, 4)
    if kind != "grid2d":
        # steps within 0.03 cells: no evaluation point changes cells
        g = np.sqrt(1.0 + (st["u"] ** 2).sum(0))
        p = dict(p, dt=0.02)
        st["dxp"] = p["dt"] * st["u"][:len(dims)] / g
        ok = np.abs(st["dxp"]).max(0) < 0.02
        assert ok.sum() > 3000
        st = inputs.subset(st, np.nonzero(ok)[0])
    got, ref, gs, _, _ = run_both(G, fields, st, p, precision="mixed", pos_mode="pair", **over)
    same = got["flags"] == ref["flags"]
    assert same.mean() > 0.995 and gs["n_nonfinite"] == 0
    d = periodic_diff(got["x"], ref["x"], [float(v) for v in dims])[:, same]
    un = np.linalg.norm(ref["u"][:, same], axis=0) + 1.0
    du = np.abs(got["u"][:, same] - ref["u"][:, same]) / un
    # reconnection's field vanishes near its null points: a few particles are
    # ill-conditioned there
    assert np.quantile(np.abs(d), 0.999) < 1e-5 and np.quantile(du, 0.999) < 1e-4


def test_axis_longer_than_the_short_floor(G):
    ny = 4
    y = np.arange(ny)[:, None]
    n = 5000
    rng = np.random.default_rng(8)
    u = rng.normal(size=(3, n))
    xs = rng.integers(0, 16 * 1024, n) / 1024.0            # exact in float32 on both axes
    ys = rng.integers(0, ny * 1024, n) / 1024.0
    out = {}
    for nx in (16, (1 << 22) + 16):
        row = np.ones((1, nx))
        Z = np.zeros((ny, nx))
        fields = dict(E=[Z, Z, 0.1 * np.cos(np.pi * y / 2) * row],
                      B=[np.sin(np.pi * y / 2) * row, Z, 1.0 + Z], dB=None, dx=(1.0, 1.0))
        # on the long axis every second particle 1024 cells on, the others at its start
        x = xs + (0.0 if nx == 16 else np.where(np.arange(n) % 2, 0.0, 1024.0))
        st = dict(x=np.stack([x, ys]), u=u, dxp=0.4 * u[:2] / np.sqrt(1 + (u ** 2).sum(0)),
                  flags=np.zeros(n, np.uint8))
        grid = G.Grid(fields, dtype="f32")
        ds = G.State.from_numpy(st, precision="mixed", pos_mode="pair")
        p = dict(qm=(50.0,), dt=0.4, dl=1.0, f_rho=0.4, grad_mode=0)
        s = G.push(ds, grid, G.make_params(p), 1)
        assert s["n_gca"] > n // 2
        out[nx] = (ds.u.cpu().numpy(), ds.dxp.cpu().numpy(), ds.flags.cpu().numpy())
    a, b = out.values()
    for p_, q in zip(a, b):
        np.testing.assert_array_equal(p_, q)
