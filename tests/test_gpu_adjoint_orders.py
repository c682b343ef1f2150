"""The adjoint with particles sorted at its checkpoints, over one to four
checkpoints (an even and an odd number of reorderings of the adjoint, which go
back and forth between the caller's arrays and scratch ones), one particle and
a ragged count, both layouts, with and without ids: each particle's arithmetic
is the unsorted one, so states, ids and state gradients are equal bit for bit;
the node gradients to the rounding of their FP64 additions (n times the points
of a step, 2^-53 each, against the largest: 1e-11)."""
import numpy as np
import pytest

from paper_2007_14401_gb300 import inputs

pytestmark = pytest.mark.gpu

STEPS = 7


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2007_14401_gb300 import gcb
    return gcb


def sweep(G, n, precision, pos_mode, gdt, ckpt, sort, fwd, pid):
    import torch
    base, pats, amps, st0, params = inputs.reconnection_2d_modes(
        nx=64, ny=32, delta=2.0, n_modes=2, max_mode=2, n_particles=1024, omega_dt_max=5.0, seed=3)
    st0 = {k: np.ascontiguousarray(v[..., :n]) for k, v in st0.items()}
    grid = G.Grid(inputs.combine_fields(base, pats, amps), dtype=gdt)
    s = G.State.from_numpy(st0, precision=precision, pos_mode=pos_mode, with_pid=pid)
    p = G.make_params(params, sort_every=sort, sort_tile=(1, 1), gca_fixed_iters=4)
    ws = G.AdjointWorkspace(s, grid, STEPS, ckpt, p)
    start = s.clone()
    stats = G.push_ckpt(s, grid, p, STEPS, ws, stats=True)
    lam = torch.randn((7, n), dtype=s.u.dtype, device="cuda",
                      generator=torch.Generator(device="cuda").manual_seed(5))
    if fwd:
        grad = G.adjoint(start, grid, p, STEPS, lam, ckpt, workspace=ws)
    else:
        grad = G.adjoint(start, grid, p, STEPS, lam, ckpt)
    return s.to_numpy(), stats, lam.cpu().numpy(), grad.cpu().numpy()


@pytest.mark.parametrize("precision,pos_mode,gdt", [("fp64", "f64", "f64"), ("mixed", "pair", "f32")])
@pytest.mark.parametrize("ckpt", [7, 4, 3, 2])
@pytest.mark.parametrize("n,fwd,pid", [(1, True, False), (1003, True, True), (1003, False, False)])
def test_orders(G, precision, pos_mode, gdt, ckpt, n, fwd, pid):
    a = sweep(G, n, precision, pos_mode, gdt, ckpt, 0, fwd, pid)
    b = sweep(G, n, precision, pos_mode, gdt, ckpt, 1, fwd, pid)
    for k in a[0]:
        np.testing.assert_array_equal(a[0][k], b[0][k], err_msg=k)
    assert all(a[1][k] == b[1][k] for k in a[1] if isinstance(a[1][k], int))
    np.testing.assert_array_equal(a[2], b[2])
    np.testing.assert_allclose(a[3], b[3], rtol=0, atol=1e-11 * np.abs(a[3]).max())
