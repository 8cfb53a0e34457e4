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


@pytest.mark.parametrize("d", [16, 20, 64])
@pytest.mark.parametrize("cap", [1, 300])
def test_cells_rescan_after_pair_overflow(kc, monkeypatch, d, cap):
    # rows whose undecided pairs do not fit the buffer are scanned against the
    # centers of their near cells
    monkeypatch.setenv("KC_EIM_CELLS", "1")
    monkeypatch.setenv("KC_TC_STREAM_CENTERS", "1")
    monkeypatch.setenv("KC_PRUNE_PAIR_CAP", str(cap))
    _check(kc, I.gauss_mixture(30_011, d, 850 + d, 30, 0.5, -10.0, 10.0, heavy_frac=0.5), 4, 850 + d)


def _timed(kc, monkeypatch, x, k, cells):
    import time

    import torch
    if cells is not None:
        monkeypatch.setenv("KC_EIM_CELLS", cells)
    else:
        monkeypatch.delenv("KC_EIM_CELLS", raising=False)
    best = float("inf")
    for _ in range(3):
        torch.cuda.synchronize()
        t = time.perf_counter()
        r = kc.kc_eim(x, k, seed=3)
        best = min(best, time.perf_counter() - t)
    return best, r.centers.cpu().tolist()


def test_cells_with_many_undecided_pairs_pay(kc, monkeypatch):
    """Half of the points in one cluster: 20M undecided pairs overflow the
    buffer.  Scanning those rows against all of S took twice the whole block's
    time; the near cells' part of it takes a third."""
    import torch
    n, d = 2_000_000, 20
    g = torch.Generator(device="cuda").manual_seed(11)
    c = torch.randint(0, 40, (n,), generator=g, device="cuda")
    c[torch.rand(n, generator=g, device="cuda") < 0.5] = 0
    x = torch.randn(n, d, generator=g, device="cuda").mul_(0.5)
    x += (20 * torch.rand(40, d, generator=g, device="cuda"))[c]
    (t, a), (t0, b) = _timed(kc, monkeypatch, x, 200, None), _timed(kc, monkeypatch, x, 200, "0")
    assert a == b
    assert t < 0.8 * t0, (t, t0)


@pytest.mark.parametrize("n,d,k", [(500_000, 12, 20), (2_000_000, 8, 25)])
def test_cells_only_where_a_sample_shows_that_they_pay(kc, monkeypatch, n, d, k):
    """Uniform points, whose cells are all near one another, take the whole
    block (by cells 1.1 to 1.3 times its time)."""
    import torch
    x = torch.rand(n, d, generator=torch.Generator(device="cuda").manual_seed(860), device="cuda")
    (t, a), (t0, b) = _timed(kc, monkeypatch, x, k, None), _timed(kc, monkeypatch, x, k, "0")
    assert a == b
    assert t < 1.07 * t0, (t, t0)


def test_cells_of_few_pivots_are_counted_too(kc, monkeypatch):
    # one cluster in four dimensions and a small S: few pivots, most cells near
    import torch
    x = torch.randn(478_764, 4, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    (t, a), (t0, b) = _timed(kc, monkeypatch, x, 12, None), _timed(kc, monkeypatch, x, 12, "0")
    assert a == b
    assert t < 1.07 * t0, (t, t0)
