"""The unit of the fields is the caller's: fields multiplied by a power of two
and q/m divided by it give the same orbits.  Every product of the step then
scales by a power of two, exactly, so that the scaled run equals the unscaled
one but for terms that leave the FP32 range on their own (and do not matter in
their sums): 1e-5 relative (100 roundings of 6e-8, twice) for 999 particles of
1000.  Scales of 8.6e9 and 1.8e13 either way, where fourth powers of the field
and third powers of its inverse are outside FP32.
"""
import numpy as np
import pytest

from paper_2007_14401_gb300 import inputs
from tests.helpers import periodic_diff

pytestmark = pytest.mark.gpu

SCALES = [-44, -33, 33, 44]
TOL = 1e-5


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2007_14401_gb300 import gcb
    return gcb


def scaled(fields, p, k):
    s = 2.0 ** k
    f = dict(fields, E=[s * np.asarray(c) for c in fields["E"]],
             B=[s * np.asarray(c) for c in fields["B"]])
    if fields.get("dB") is not None:
        f["dB"] = [s * np.asarray(c) for c in fields["dB"]]
    return f, dict(p, qm=tuple(q / s for q in p["qm"]))


def case(kind):
    if kind == "grid2d":
        return inputs.reconnection_2d(nx=64, ny=32, n_particles=4001, seed=9) + ((64.0, 32.0),)
    if kind == "dw2d":
        f, st, p = inputs.harris_2d(n_per_species=1001, seed=9)
        return f, st, p, (128.0, 128.0)
    return inputs.current_sheet_3d(n=24, n_particles=4001, seed=9) + ((24.0,) * 3,)


@pytest.mark.parametrize("k", SCALES)
@pytest.mark.parametrize("kind", ["grid2d", "dw2d", "dw3d"])
@pytest.mark.parametrize("option", ["plain", "mirror", "uperp", "no curvature"])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_push(G, kind, option, precision, k):
    fields, st, p, L = case(kind)
    over = {"plain": {}, "mirror": dict(mirror=1), "uperp": dict(mu_mode=1),
            "no curvature": dict(curvature=0)}[option]
    res = []
    for kk in (0, k):
        f, q = scaled(fields, p, kk)
        grid = G.Grid(f, dtype="f64" if precision == "fp64" else "f32")
        ds = G.State.from_numpy(st, precision=precision, pos_mode="pair")
        s = G.push(ds, grid, G.make_params(q, gca_fixed_iters=5, **over), 2)
        res.append((ds.to_numpy(), s))
    (a, sa), (b, sb) = res
    assert sa["n_gca"] > 0.2 * a["flags"].size
    for key in ("n_gca", "n_boris", "n_gcafail", "n_nonfinite"):
        assert abs(sa[key] - sb[key]) <= 2e-3 * a["flags"].size, key
    bad = a["flags"] != b["flags"]
    bad |= (np.abs(periodic_diff(a["x"], b["x"], L)) > TOL).any(0)
    bad |= (np.abs(a["u"] - b["u"]) > TOL * (1.0 + np.linalg.norm(a["u"], axis=0))).any(0)
    bad |= (np.abs(a["dxp"] - b["dxp"]) > TOL).any(0)
    assert bad.mean() < 1e-3


@pytest.mark.parametrize("k", SCALES)
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_adjoint(G, precision, k):
    """Gradients of the state as they are, those of the records by 2^-k."""
    import torch
    base, pats, amps, st, p = inputs.reconnection_2d_modes(
        nx=64, ny=32, delta=2.0, n_modes=2, max_mode=2, n_particles=2003, omega_dt_max=50.0, seed=3)
    fields = inputs.combine_fields(base, pats, amps)
    res = []
    for kk in (0, k):
        f, q = scaled(fields, p, kk)
        grid = G.Grid(f, dtype="f64" if precision == "fp64" else "f32")
        ds = G.State.from_numpy(st, precision=precision, pos_mode="pair")
        lam = torch.randn((7, ds.n), dtype=ds.u.dtype, device="cuda",
                          generator=torch.Generator(device="cuda").manual_seed(5))
        grad = G.adjoint(ds, grid, G.make_params(q, gca_fixed_iters=4), 2, lam, 2)
        res.append((lam.double().cpu().numpy(), grad.cpu().numpy() * 2.0 ** kk))
    for a, b in zip(*res):
        ref = a if a.shape[0] == 7 else a.T
        got = b if b.shape[0] == 7 else b.T
        rms = np.sqrt((ref ** 2).mean(1, keepdims=True))
        assert (rms > 0).all() and np.isfinite(got).all()
        assert (np.abs(got - ref) > TOL * (np.abs(ref) + rms)).mean() < 1e-3
