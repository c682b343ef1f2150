"""Pushes without statistics run kernels of their own: every particle comes out
as from the call with statistics, bit for bit, on each path (precisions,
options, deposition, several steps a launch, covariant); and a program that has
only pushed with statistics can capture pushes into a graph."""
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


def same(a, b):
    for k in ("x", "u", "dxp", "flags"):
        np.testing.assert_array_equal(a[k], b[k])


@pytest.mark.parametrize("field", ["recon", "sheet", "harris"])
@pytest.mark.parametrize("precision,pos_mode", [("fp64", "f64"), ("mixed", "pair"), ("mixed", "f64")])
@pytest.mark.parametrize("option", ["plain", "fuse", "exact", "mirror", "deposit"])
def test_same_particles(G, field, precision, pos_mode, option):
    if field == "recon":
        fields, st, p = inputs.reconnection_2d(nx=64, ny=32, n_particles=3001, seed=6)
    elif field == "sheet":
        fields, st, p = inputs.current_sheet_3d(n=24, n_particles=3001, seed=6)
    else:
        fields, st, p = inputs.harris_2d(n_per_species=701, seed=6)
    if option == "exact" and (precision, pos_mode) == ("mixed", "f64"):
        pytest.skip("the exact frame has no kernels for this layout")
    st["u"][0, 5] = np.nan                      # one frozen particle
    over = dict(plain={}, fuse=dict(fuse_steps=3), exact=dict(drift_frame=1),
                mirror=dict(mirror=1), deposit={})[option]
    res = []
    for stats in (True, False):
        grid = G.Grid(fields, dtype="f64" if precision == "fp64" else "f32")
        ds = G.State.from_numpy(st, precision=precision, pos_mode=pos_mode)
        cur = G.Current(grid, (1.0, -1.0, 1.0, -1.0), precision) if option == "deposit" else None
        out = G.push(ds, grid, G.make_params(p, **over), 3, stats=stats, current=cur)
        assert (out is None) == (not stats)
        res.append(ds.to_numpy())
    same(*res)


def test_same_particles_covariant(G):
    fields, st, p = inputs.kerr_wald(nr=64, nth=48, n_particles=3001, seed=6)
    res = []
    for stats in (True, False):
        grid = G.KsGrid(fields, p["a"], p["r_in"], p["r_out"])
        ds = G.State.from_numpy(st, precision="fp64")
        G.push_ks(ds, grid, G.make_params(p), 3, stats=stats)
        res.append(ds.to_numpy())
    same(*res)


def test_capture_after_a_push_with_statistics(G):
    fields, st, p = inputs.reconnection_2d(nx=64, ny=32, n_particles=3001, seed=7)
    res = []
    for graphed in (True, False):
        grid = G.Grid(fields, dtype="f32")
        ds = G.State.from_numpy(st, precision="mixed", pos_mode="pair")
        gp = G.make_params(p)
        ws = G.Workspace(ds, grid, gp)
        G.push(ds, grid, gp, 1, workspace=ws, stats=True)
        if graphed:
            G.StepGraph(ds, grid, gp, 4, ws).replay()
        else:
            G.push(ds, grid, gp, 4, workspace=ws, stats=False)
        res.append(ds.to_numpy())
    same(*res)
