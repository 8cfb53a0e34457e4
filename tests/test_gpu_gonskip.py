"""The Gonzalez steps that leave out distances by the triangle inequality
(KC_GON_SKIP=1 changes over at the first probe, after 16 steps) against the
oracle: sizes around units of 32 and blocks of 128 points, several regroupings,
coordinate counts around the loads' batches, unaligned rows, ties, duplicate
points and an early stop, and behind the low-precision sweeps.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1604_03228_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _check(kc, pts, k, first=0, **kw):
    x = kw.pop("x", None)
    r = kc.kc_gonzalez(_dev(pts) if x is None else x, k, first=first, **kw)
    ref = O.gonzalez(pts, k, first=first, mode="f32")
    assert r.centers.cpu().numpy().tolist() == ref.centers.tolist()
    assert r.k_out == len(ref.centers)
    assert r.radius == O.radius(pts, ref.centers, mode="f64")[0]


@pytest.fixture(autouse=True)
def _forced(monkeypatch):
    monkeypatch.setenv("KC_GON_SKIP", "1")
    monkeypatch.setenv("KC_GON_RESIDENT", "0")


@pytest.mark.parametrize("n,d,k", [(31, 3, 30), (129, 5, 60), (4097, 1, 40), (20_000, 16, 200), (33_333, 37, 100),
                                   (60_000, 64, 300), (9_000, 65, 40), (5_000, 130, 30), (50_000, 2, 600)])
@pytest.mark.parametrize("shape", ["gau", "unif"])
def test_skip_equals_oracle(kc, n, d, k, shape):
    pts = (I.gauss_mixture(n, d, 700 + d, 20, 0.5, -10.0, 10.0) if shape == "gau" else I.unif_points(n, d, 700 + d))
    _check(kc, pts, k, first=n // 3)


@pytest.mark.parametrize("n,d,k", [(4_000, 256, 40), (4_000, 257, 40), (3_000, 768, 30), (3_000, 769, 30),
                                   (2_500, 1100, 70), (1_500, 3700, 30)])
def test_skip_large_d(kc, n, d, k):
    # the assignment stages centers in parts of 256 coordinates
    _check(kc, I.gauss_mixture(n, d, 720 + d, 20, 0.5, -10.0, 10.0), k, first=5)


@pytest.mark.parametrize("sweep", ["f32", "bf16"])
@pytest.mark.parametrize("shape", ["gau", "unif"])
def test_skip_large_d_with_the_default_switches(kc, monkeypatch, shape, sweep):
    # large enough for the segments by itself (n d k >= 1e10): the same as the
    # streaming kernels, whether it changes over or not
    import torch
    n, d, k = 200_000, 1024, 64
    g = torch.Generator(device="cuda").manual_seed(730)
    x = torch.randn(n, d, generator=g, device="cuda")
    if shape == "gau":
        x += 20.0 * torch.rand(10, d, generator=g, device="cuda")[torch.randint(0, 10, (n,), generator=g, device="cuda")]
    monkeypatch.delenv("KC_GON_SKIP")
    a = kc.kc_gonzalez(x, k, sweep=sweep)
    monkeypatch.setenv("KC_GON_SKIP", "0")
    b = kc.kc_gonzalez(x, k, sweep=sweep)
    assert a.centers.cpu().tolist() == b.centers.cpu().tolist() and (a.k_out, a.radius) == (b.k_out, b.radius)
    assert kc.kc_radius(x, a.centers).radius == a.radius


@pytest.mark.parametrize("sweep", ["bf16", "fp16", "fp8"])
def test_skip_behind_a_low_precision_sweep(kc, sweep):
    _check(kc, I.gauss_mixture(40_000, 24, 710, 30, 0.5, -10.0, 10.0), 120, sweep=sweep)


def test_skip_unaligned_rows(kc):
    import torch
    pts = I.gauss_mixture(20_000, 12, 711, 10, 0.5, -10.0, 10.0)
    buf = torch.empty(pts.size + 1, dtype=torch.float32, device="cuda")
    x = buf[1:].view(pts.shape)
    x.copy_(torch.from_numpy(pts))
    _check(kc, pts, 90, x=x)


@pytest.mark.parametrize("sweep", ["f32", "bf16"])
def test_skip_host_points(kc, sweep):
    # pinned points are copied to the device rather than read in place
    import torch
    pts = I.gauss_mixture(30_001, 9, 714, 12, 0.5, -10.0, 10.0)
    ref = O.gonzalez(pts, 300, mode="f32")
    for x in (torch.from_numpy(pts).pin_memory(), torch.from_numpy(pts), pts):
        r = kc.kc_gonzalez(x, 300, sweep=sweep)
        assert np.asarray(r.centers).tolist() == ref.centers.tolist()
        assert r.radius == O.radius(pts, ref.centers, mode="f64")[0]


def test_skip_ties_duplicates_and_early_stop(kc):
    grid = I.int_points(30_000, 3, 712, 0, 4).astype(np.float32)   # 125 distinct points
    _check(kc, grid, 100)
    r = kc.kc_gonzalez(_dev(grid), 300)
    assert r.k_out == len(O.gonzalez(grid, 300, mode="f32").centers) < 300 and r.radius == 0.0


@pytest.mark.parametrize("scale", [1e-22, 2e-20, 1e-15, 1e16])
def test_skip_tiny_and_huge_coordinates(kc, monkeypatch, scale):
    # squared distances that underflow, and near the largest accepted
    # magnitude: the same as the streaming kernel
    pts = (I.gauss_mixture(20_000, 4, 713, 8, 0.01, -1.0, 1.0) * np.float32(scale)).astype(np.float32)
    x = _dev(pts)
    a = kc.kc_gonzalez(x, 60)
    monkeypatch.setenv("KC_GON_SKIP", "0")
    b = kc.kc_gonzalez(x, 60)
    assert a.centers.cpu().tolist() == b.centers.cpu().tolist() == O.gonzalez(pts, 60, mode="f32").centers.tolist()
    assert (a.k_out, a.radius) == (b.k_out, b.radius)


@pytest.mark.parametrize("kind", ["gau", "dup", "unaligned", "host"])
def test_skip_on_eims_sample_equals_oracle(kc, kind):
    # the rows of the sample are found through its index
    import torch
    n, d, k = 40_009, 9, 24
    pts = I.gauss_mixture(n, d, 750, 15, 0.5, -10.0, 10.0)
    if kind == "dup":
        pts = np.ascontiguousarray(pts[np.arange(n) % 20_000])
    x = pts
    if kind == "unaligned":
        x = torch.empty(pts.size + 1, dtype=torch.float32, device="cuda")[1:].view(pts.shape)
        x.copy_(torch.from_numpy(pts))
    elif kind != "host":
        x = _dev(pts)
    r = kc.kc_eim(x, k, eps=0.1, phi=6.0, seed=7)
    ref = O.eim(pts, k, 0.1, 6.0, 7, mode="f32")
    assert np.asarray(r.centers if kind == "host" else r.centers.cpu()).tolist() == ref.centers.tolist()
    assert r.radius == O.radius(pts, ref.centers, mode="f64")[0]


@pytest.mark.parametrize("n,d,k", [(800_000, 12, 200), (60_000, 1000, 30), (1_500_001, 33, 300)])
def test_skip_on_eims_sample_equals_streaming(kc, monkeypatch, n, d, k):
    import torch
    g = torch.Generator(device="cuda").manual_seed(751)
    x = torch.randn(n, d, generator=g, device="cuda").mul_(0.5)
    x += (20.0 * torch.rand(40, d, generator=g, device="cuda"))[torch.randint(0, 40, (n,), generator=g, device="cuda")]
    a = kc.kc_eim(x, k, seed=3)
    monkeypatch.setenv("KC_GON_SKIP", "0")
    b = kc.kc_eim(x, k, seed=3)
    assert a.centers.cpu().tolist() == b.centers.cpu().tolist() and (a.k_out, a.radius) == (b.k_out, b.radius)


@pytest.mark.parametrize("n,d,k,clusters,gain", [(10_000_000, 8, 500, 0, 0.0), (10_000_000, 10, 1024, 1, 0.0),
                                                 (4_000_000, 16, 512, 40, 0.5)])
def test_probe_changes_over_only_where_it_pays(kc, monkeypatch, n, d, k, clusters, gain):
    """Points without clusters stay on the streaming kernel (two of the slowest
    mistakes took 2.0 and 2.1 times as long), clustered ones leave it."""
    import time

    import torch
    g = torch.Generator(device="cuda").manual_seed(740)
    if clusters:
        x = torch.randn(n, d, generator=g, device="cuda").mul_(0.5)
        x += (20.0 * torch.rand(clusters, d, generator=g, device="cuda"))[torch.randint(0, clusters, (n,), generator=g, device="cuda")]
    else:
        x = torch.rand(n, d, generator=g, device="cuda")

    def solve(switch):
        if switch:
            monkeypatch.setenv("KC_GON_SKIP", switch)
        else:
            monkeypatch.delenv("KC_GON_SKIP")
        best = float("inf")
        for _ in range(4):
            torch.cuda.synchronize()
            t = time.perf_counter()
            r = kc.kc_gonzalez(x, k)
            best = min(best, time.perf_counter() - t)
        return best, r.centers.cpu().tolist()

    (t, c), (t0, c0) = solve(None), solve("0")
    assert c == c0
    assert t < (1.0 - gain if gain else 1.25) * t0, (t, t0)
