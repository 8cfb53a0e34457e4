"""EIM's prune by Voronoi cells (KC_EIM_CELLS=1 takes it wherever S has 1024
points) against the oracle: the CUDA-core path at coordinate counts around its
specialisations, the tensor-core path at its smallest and largest d, clustered
and uniform points, duplicates, and unaligned rows; and a large case against
the whole block."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1604_03228_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _check(kc, pts, k, seed, x=None):
    r = kc.kc_eim(_dev(pts) if x is None else x, k, eps=0.1, phi=6.0, seed=seed)
    ref = O.eim(pts, k, 0.1, 6.0, seed, mode="f32")
    assert r.centers.cpu().numpy().tolist() == ref.centers.tolist()
    assert r.radius == O.radius(pts, ref.centers, mode="f64")[0]


@pytest.mark.parametrize("d", [1, 2, 3, 5, 9, 15, 16, 33, 64, 93, 94])
@pytest.mark.parametrize("shape", ["gau", "unif"])
def test_cells_equal_oracle(kc, monkeypatch, d, shape):
    monkeypatch.setenv("KC_EIM_CELLS", "1")
    if d >= 16:   # few centers would stay in shared memory and take no cells
        monkeypatch.setenv("KC_TC_STREAM_CENTERS", "1")
    n = 30_011
    pts = (I.gauss_mixture(n, d, 800 + d, 30, 0.5, -10.0, 10.0) if shape == "gau" else I.unif_points(n, d, 800 + d))
    _check(kc, pts, 4, 800 + d)


def test_cells_duplicates_and_unaligned_rows(kc, monkeypatch):
    import torch
    monkeypatch.setenv("KC_EIM_CELLS", "1")
    _check(kc, I.int_points(40_000, 3, 830, 0, 9).astype(np.float32), 4, 1)   # 1000 distinct points
    pts = I.gauss_mixture(30_000, 20, 831, 10, 0.5, -10.0, 10.0)
    buf = torch.empty(pts.size + 1, dtype=torch.float32, device="cuda")
    x = buf[1:].view(pts.shape)
    x.copy_(torch.from_numpy(pts))
    _check(kc, pts, 4, 2, x)


@pytest.mark.parametrize("n,d,k", [(1_000_000, 2, 50), (600_000, 64, 40)])
def test_cells_equal_the_whole_block(kc, monkeypatch, n, d, k):
    x = _dev(I.gauss_mixture(n, d, 840 + d, 40, 0.5, -10.0, 10.0))
    got = []
    for v in ("1", "0"):
        monkeypatch.setenv("KC_EIM_CELLS", v)
        r = kc.kc_eim(x, k, seed=3)
        got.append((r.centers.cpu().tolist(), r.radius))
    assert got[0] == got[1]
