"""FP32-pair positions are sorted as pairs: a particle whose low part alone is
not finite goes last, as every particle with a non-finite position does."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2007_14401_gb300 import gcb
    return gcb


@pytest.mark.parametrize("nd", [2, 3])
@pytest.mark.parametrize("n", [40, 5003])
def test_non_finite_low_part_last(G, nd, n):
    shape = (16,) * nd
    rng = np.random.default_rng(n)
    fields = dict(E=[np.zeros(shape)] * 3, B=[np.zeros(shape)] * 3, dB=None, dx=(1.0,) * nd)
    grid = G.Grid(fields, dtype="f32")
    st = dict(x=rng.uniform(0.0, 16.0, (nd, n)), u=np.zeros((3, n)), dxp=np.zeros((nd, n)),
              flags=np.zeros(n, np.uint8))
    ds = G.State.from_numpy(st, precision="mixed", pos_mode="pair", with_pid=True)
    bad = {3: np.nan, 17: np.inf, n - 2: -np.inf, n // 2: np.nan}
    for i, v in bad.items():
        ds.x_lo[i % nd, i] = v
    G.sort(ds, grid, G.make_params(dict(qm=(1.0,), dt=0.1), sort_every=1, sort_tile=(1,) * nd))
    pid = ds.pid.cpu().numpy()
    assert sorted(pid[-len(bad):]) == sorted(bad)
    x = ds.x.cpu().numpy()[:, :-len(bad)]
    key = np.zeros(x.shape[1], int)
    for d in reversed(range(nd)):
        key = key * 16 + np.floor(x[d]).astype(int).clip(0, 15)
    assert (np.diff(key) >= 0).all()
