"""The sort at the sizes where its kernels' pieces end: particle counts around
a warp and a block's four items a thread, runs of one cell longer than a warp
and none at all, 2D and 3D, both position forms, and a grid with more chunks
of cells than each block of the scan adds up itself."""
import numpy as np
import pytest

from tests.test_gpu_sort import tile_key

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2007_14401_gb300 import gcb
    return gcb


def check(G, shape, x, pos_mode, precision="mixed"):
    nd, n = x.shape
    dims = tuple(reversed(shape))
    row = np.zeros(shape)
    fields = dict(E=[row] * 3, B=[row] * 3, dB=None, dx=(1.0,) * nd)
    grid = G.Grid(fields, dtype="f64" if precision == "fp64" else "f32")
    st = dict(x=x, u=np.arange(3.0 * n).reshape(3, n) % 1021, dxp=np.arange(nd * n).reshape(nd, n) % 509,
              flags=(np.arange(n) % 4 << 6).astype(np.uint8))
    ds = G.State.from_numpy(st, precision=precision, pos_mode=pos_mode, with_pid=True)
    gp = G.make_params(dict(qm=(1.0,), dt=0.1), sort_every=1, sort_tile=(1,) * nd)
    before = ds.to_numpy()
    G.sort(ds, grid, gp)
    after = ds.to_numpy()
    pid = after["pid"]
    assert np.array_equal(np.sort(pid), np.arange(n))
    for k in ("x", "u", "dxp", "flags"):
        assert np.array_equal(after[k], before[k][..., pid], equal_nan=(k != "flags"))
    fin = np.isfinite(after["x"]).all(0)
    # the cell in FP32, as the sort takes it (within rounding of a face either side)
    x32 = after["x"][:, fin].astype(np.float32).astype(np.float64)
    key = tile_key(x32, (1.0,) * nd, dims, (1,) * nd)
    assert np.all(np.diff(key) >= 0)
    assert fin[:int(fin.sum())].all()          # non-finite positions last


@pytest.mark.parametrize("n", [1, 31, 33, 255, 1023, 1024, 1025, 70001])
@pytest.mark.parametrize("nd,precision,pos_mode", [(2, "mixed", "pair"), (3, "mixed", "pair"),
                                                   (2, "mixed", "f64"), (3, "fp64", "f64")])
def test_counts(G, n, nd, precision, pos_mode):
    shape = (37, 64) if nd == 2 else (9, 17, 32)
    dims = np.array(tuple(reversed(shape)), dtype=float)[:, None]
    rng = np.random.default_rng(n)
    for kind in ("random", "one cell", "pairs"):
        x = rng.uniform(0.0, 1.0, (nd, n)) * dims
        if kind == "one cell":
            x = 3.25 + 0.5 * rng.uniform(0.0, 1.0, (nd, n))
        elif kind == "pairs":
            x = np.floor(x[:, np.arange(n) // 2]) + 0.5
        if n > 40:
            x[0, 7], x[1, 39] = np.nan, np.inf
        check(G, shape, x, pos_mode, precision)


def test_more_chunks_than_each_block_adds_up(G):
    shape = (4200, 8192)                       # 8400 chunks of 4096 cells
    rng = np.random.default_rng(5)
    x = rng.uniform(0.0, 1.0, (2, 100003)) * np.array([[8192.0], [4200.0]])
    check(G, shape, x, "pair")
