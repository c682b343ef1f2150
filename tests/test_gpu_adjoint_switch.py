"""The adjoint transposes the branch that the forward run took, also for
particles within rounding of the switch's threshold: the gradient of each is,
bit for bit, that of the run forced onto the branch its flag names."""
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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("method", ["reverse", "tangent"])
@pytest.mark.parametrize("where", ["nodes", "anywhere"])
def test_branch_at_the_threshold(G, precision, method, where):
    import torch
    n, nx, ny = 20000, 16, 8
    one = np.ones((ny, nx))
    # Gamma = f_rho dl |q/m| B to a few roundings, any direction
    b, q = 1.3, 5.0
    eps = 2.2e-16 if precision == "fp64" else 1.2e-7
    rng = np.random.default_rng(4)
    d = rng.normal(size=(3, n))
    d /= np.linalg.norm(d, axis=0)
    u = d * np.sqrt((0.4 * q * b) ** 2 - 1.0) * (1.0 + rng.integers(-6, 7, n) * eps)
    x = np.stack([rng.uniform(0, nx, n), rng.uniform(0, ny, n)])
    st = dict(x=np.floor(x) if where == "nodes" else x, u=u, dxp=0.1 * u[:2],
              flags=np.zeros(n, np.uint8))
    B = [0.3 * b * one, 0.4 * b * one, np.sqrt(0.75) * b * one]
    fields = dict(E=[0.0 * one, 0.0 * one, 0.01 * one], B=B,
                  dB=inputs.central_gradients(B, (1.0, 1.0)), dx=(1.0, 1.0))
    grid = G.Grid(fields, dtype="f64" if precision == "fp64" else "f32")
    lam0 = torch.randn((7, n), dtype=torch.float64, device="cuda",
                       generator=torch.Generator(device="cuda").manual_seed(1))
    out, S = {}, None
    for force in (0, 1, 2):
        gp = G.make_params(dict(qm=(q,), dt=0.3), grad_mode=1, gca_fixed_iters=3, force=force)
        ds = G.State.from_numpy(st, precision=precision, pos_mode="pair")
        ws = G.AdjointWorkspace(ds, grid, 1, 1, gp)
        start = ds.clone()
        G.push_ckpt(ds, grid, gp, 1, ws)
        if force == 0:
            S = ds.flags.cpu().numpy() & 1
        lam = lam0.to(ds.u.dtype).clone()
        G.adjoint(start, grid, gp, 1, lam, 1, method=method, workspace=ws)
        out[force] = lam.cpu().numpy()
    assert 0.1 < S.mean() < 0.9
    assert (out[1] != out[2]).any(0).all()
    np.testing.assert_array_equal(out[0], np.where(S, out[1], out[2]))
