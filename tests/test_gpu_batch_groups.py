"""The batched form's CTA groups: instances side by side, and groups that solve
several instances one after another, against the plain queue on the same
batch (every instance) and the oracle (some): block and warp remainders, all
d loops of the mixed launch, k at and above n, early stops, and a batch whose
exchange slots would take too much scratch.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1604_03228_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SIZES = (1, 31, 128, 129, 1000, 1024, 1025, 2047, 5000, 20_001)


def _batch(count, dims, big, integer, seed):
    insts, ks = [], []
    for i in range(count):
        n, d = SIZES[i % len(SIZES)], dims[(i // 3) % len(dims)]
        if i < big:
            n = 60_000 + 131 * i
        if integer:
            p = I.int_points(n, d, seed + i, -500, 500)
        else:
            p = I.gauss_mixture(n, d, seed + i, 7, 0.2, 0, 1)
        if i % 11 == 5:
            p = np.ascontiguousarray(p[np.arange(n) % min(n, 9)])   # nine distinct points
        insts.append(p)
        ks.append((1, 7, 33, 64, 130)[i % 5])
    return insts, ks


@pytest.mark.parametrize("count,big", [(9, 2), (700, 3)])
@pytest.mark.parametrize("sweep,dims", [("f32", (2, 3, 8, 16, 32, 37)), ("f32", (8,)), ("bf16", (3, 5, 8, 32)),
                                        ("bf16", (32,)), ("int", (2, 7))])
def test_batch_groups_match_queue(kc, monkeypatch, count, big, sweep, dims):
    import torch
    insts, ks = _batch(count, dims, big, sweep == "int", 7000 + count)
    xs = [torch.from_numpy(p).cuda() for p in insts]
    kw = {} if sweep == "int" else {"sweep": sweep}
    plan = kc.kc_batch_plan_create(xs, ks, **kw)
    theta, nheavy, gheavy, grid = kc.kc_batch_plan_info(plan)
    assert theta == 1.0 and nheavy >= big and gheavy <= grid
    assert (count > grid) == (count == 700)     # more instances than fit side by side
    for _ in range(2):
        kc.kc_batch_plan_run(plan)
        got = kc.kc_batch_plan_wait(plan)
    got = [(r.centers.cpu().tolist(), r.k_out, r.radius) for r in got]
    kc.kc_batch_plan_destroy(plan)
    call = kc.kc_gonzalez_batch(xs, ks, **kw)
    assert [(r.centers.cpu().tolist(), r.k_out, r.radius) for r in call] == got
    monkeypatch.setenv("KC_BATCH_THETA", "inf")
    ref = kc.kc_gonzalez_batch(xs, ks, **kw)
    assert [(r.centers.cpu().tolist(), r.k_out, r.radius) for r in ref] == got
    for i in range(min(count, 12)):
        o = O.gonzalez(insts[i], ks[i], mode="i64" if sweep == "int" else "f32")
        assert got[i][0] == o.centers.tolist()


@pytest.mark.parametrize("sweep", ["f32", "bf16"])
def test_batch_groups_keep_scratch(kc, monkeypatch, sweep):
    """k = n: the slots of 700 groups would take more scratch than the points."""
    import torch
    xs = [torch.from_numpy(I.gauss_mixture(1500, 3, 90 + i, 5, 0.2, 0, 1)).cuda() for i in range(900)]
    ks = [1500] * len(xs)
    plan = kc.kc_batch_plan_create(xs, ks, sweep=sweep)
    nheavy = kc.kc_batch_plan_info(plan)[1]
    kc.kc_batch_plan_run(plan)
    got = [(r.centers.cpu().tolist(), r.k_out, r.radius) for r in kc.kc_batch_plan_wait(plan)]
    kc.kc_batch_plan_destroy(plan)
    monkeypatch.setenv("KC_BATCH_THETA", "1")
    plan = kc.kc_batch_plan_create(xs, ks, sweep=sweep)
    assert kc.kc_batch_plan_info(plan)[1] == nheavy
    kc.kc_batch_plan_run(plan)
    assert [(r.centers.cpu().tolist(), r.k_out, r.radius) for r in kc.kc_batch_plan_wait(plan)] == got
    kc.kc_batch_plan_destroy(plan)


@pytest.mark.parametrize("d,integer", [(2, False), (10, False), (16, False), (24, False), (100, False), (7, True), (64, True)])
def test_one_d_batches_keep_four_ctas_per_sm(kc, d, integer):
    """A batch of one d has a kernel of its own, not the one of several d with
    its loops out of line (128 registers a thread): as many CTAs as at d = 8."""
    import torch

    def solve(dd):
        make = (lambda i: I.int_points(200, dd, 60 + i, -99, 99)) if integer else (lambda i: I.gauss_mixture(200, dd, 60 + i, 5, 0.2, 0, 1))
        pts = [make(i % 7) for i in range(2000)]
        plan = kc.kc_batch_plan_create([torch.from_numpy(p).cuda() for p in pts], [9] * len(pts))
        grid = kc.kc_batch_plan_info(plan)[3]
        kc.kc_batch_plan_run(plan)
        got = [r.centers.cpu().tolist() for r in kc.kc_batch_plan_wait(plan)]
        kc.kc_batch_plan_destroy(plan)
        assert got[:7] == [O.gonzalez(p, 9, mode="i64" if integer else "f32").centers.tolist() for p in pts[:7]]
        assert all(g == got[i % 7] for i, g in enumerate(got))
        return grid

    assert solve(d) == solve(8)


@pytest.mark.parametrize("integer,d", [(False, 10), (False, 24), (False, 25), (False, 64), (False, 95), (False, 96),
                                       (False, 130), (True, 47), (True, 48)])
def test_one_d_batch_groups_match_queue(kc, monkeypatch, integer, d):
    """Around the lines between the kernels (d = 24 and 96) and of the grouping
    by L2 (96, int32 48)."""
    import torch
    insts, ks = _batch(700, (d,), 3, integer, 7100 + d)
    xs = [torch.from_numpy(p).cuda() for p in insts]
    got = [(r.centers.cpu().tolist(), r.k_out, r.radius) for r in kc.kc_gonzalez_batch(xs, ks)]
    monkeypatch.setenv("KC_BATCH_THETA", "inf")
    assert [(r.centers.cpu().tolist(), r.k_out, r.radius) for r in kc.kc_gonzalez_batch(xs, ks)] == got
    for i in range(11):
        o = O.gonzalez(insts[i], ks[i], mode="i64" if integer else "f32")
        assert got[i][0] == o.centers.tolist()
