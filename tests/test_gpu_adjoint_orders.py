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


@pytest.mark.parametrize("precision,pos_mode,gdt", [("mixed", "pair", "f32"), ("mixed", "f64", "f32"),
                                                    ("fp64", "f64", "f64")])
@pytest.mark.parametrize("sort", [0, 1])
def test_same_run_with_and_without_forward_checkpoints(G, precision, pos_mode, gdt, sort):
    """Without checkpoints from the forward the adjoint runs its own: both modes
    return the same run's final state, and its gradients, bit for bit."""
    import torch
    base, pats, amps, st0, params = inputs.reconnection_2d_modes(
        nx=64, ny=32, delta=2.0, n_modes=2, max_mode=2, n_particles=2003, omega_dt_max=50.0, seed=3)
    dev, n = "cuda", st0["flags"].size
    base_rec = G.Grid(base, dtype=gdt).rec
    pat_rec = torch.stack([G.Grid(p, dtype=gdt).rec for p in pats]).contiguous()
    mdt = torch.float64 if precision == "fp64" else torch.float32
    gen = torch.Generator(device=dev).manual_seed(5)
    w = [torch.randn((k, n), dtype=torch.float64, device=dev, generator=gen) for k in (2, 3, 2)]
    res = []
    for fwd in (True, False):
        grid = G.Grid(inputs.combine_fields(base, pats, amps), dtype=gdt)
        leaves = [torch.tensor(st0["x"], dtype=torch.float64, device=dev, requires_grad=True),
                  torch.tensor(st0["u"], dtype=mdt, device=dev, requires_grad=True),
                  torch.tensor(st0["dxp"], dtype=mdt, device=dev, requires_grad=True),
                  torch.tensor(amps, dtype=torch.float64, device=dev, requires_grad=True)]
        cfg = dict(grid=grid, base=base_rec, pat=pat_rec,
                   params=G.make_params(params, sort_every=sort, sort_tile=(1, 1), gca_fixed_iters=4),
                   n_steps=STEPS, ckpt_every=3, flags=torch.tensor(st0["flags"], device=dev),
                   precision=precision, pos_mode=pos_mode, ckpt_in_forward=fwd)
        out = G.ModePush.apply(*leaves, cfg)
        sum((a.double() * b).sum() for a, b in zip(out, w)).backward()
        res.append([t.detach().cpu().numpy() for t in out] + [t.grad.cpu().numpy() for t in leaves])
    a, b = res
    for x, y in zip(a[:6], b[:6]):
        np.testing.assert_array_equal(x, y)
    np.testing.assert_allclose(a[6], b[6], rtol=0, atol=1e-11 * np.abs(a[6]).max())
