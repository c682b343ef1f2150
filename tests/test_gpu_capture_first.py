"""What a program must have called before it may capture pushes into a graph:
one call with statistics readies every kernel that the same call without them
launches.  Each case in a process of its own, where no other call has readied
any.  A kernel is readied by the library's one occupancy query for it: the call
without statistics must make none, and then captures and replays."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROG = r"""
import sys
import torch
from torch.profiler import profile, ProfilerActivity
from paper_2007_14401_gb300 import gcb as G, inputs
kind, prec, part = sys.argv[1:4]
fields, st, p = inputs.reconnection_2d(nx=64, ny=32, n_particles=3001, seed=7)
p = dict(p, gca_max_iter=8)
grid = G.Grid(fields, dtype="f64" if prec == "fp64" else "f32")
ds = G.State.from_numpy(st, precision=prec, pos_mode="pair")
ref = ds.clone()
if kind == "ckpt":
    gp = G.make_params(p)
    ws = G.AdjointWorkspace(ds, grid, 4, 2, gp)
    call = lambda s, stats: G.push_ckpt(s, grid, gp, 4, ws, stats=stats)
else:
    gp = G.make_params(p, fuse_steps=4 if kind == "fuse" else 0,
                       mirror=1 if kind == "mirror" else 0)
    ws = G.Workspace(ds, grid, gp)
    call = lambda s, stats: G.push(s, grid, gp, 5, workspace=ws, stats=stats)
if part == "queries":
    def calls(f):
        with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as pr:
            f()
            torch.cuda.synchronize()
        return [e.name() for e in pr.profiler.kineto_results.events()]
    for _ in range(2):                 # a first profile may be empty
        calls(lambda: torch.ones(1024, device="cuda").add_(1))
    names = calls(lambda: call(ds, True))
    assert any("Occupancy" in n for n in names), names     # the profile shows them
    names = calls(lambda: call(ds, False))
    assert any("k_push_sr" in n for n in names), names
    assert not any("Occupancy" in n for n in names), names
    print("done")
    sys.exit(0)
call(ds, True)
call(ref, True)
torch.cuda.synchronize()
side = torch.cuda.Stream()
side.wait_stream(torch.cuda.current_stream())
g = torch.cuda.CUDAGraph()
with torch.cuda.stream(side):
    with torch.cuda.graph(g, stream=side):
        call(ds, False)
torch.cuda.current_stream().wait_stream(side)
g.replay()
torch.cuda.synchronize()
call(ref, False)
torch.cuda.synchronize()
assert torch.equal(ds.u, ref.u) and torch.equal(ds.x, ref.x) and torch.equal(ds.flags, ref.flags)
print("done")
"""


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("kind", ["plain", "fuse", "mirror", "ckpt"])
@pytest.mark.parametrize("part", ["queries", "capture"])
def test_first_call_readies_all(kind, prec, part):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", PROG, kind, prec, part], cwd=ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout + r.stderr
