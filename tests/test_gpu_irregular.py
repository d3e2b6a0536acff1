"""Rows far from what the newer routes are made for: the results, and that a call is not much slower than on the routes that do not
depend on how the timestamps fall."""
import numpy as np
import pytest
import torch

import oracle as o

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2001_01347_b200 as zl


def rows(kind, n, R, B):
    rng = np.random.default_rng(len(kind) + n)
    if kind == "standing still":                                   # one timestamp everywhere
        ts = np.full((B, n, R), 77_777)
    elif kind == "standing still for long":
        ts = np.cumsum(np.where(rng.random((B, n, R)) < 0.01, 1_000_000, 0) + (np.arange(R) == 0), axis=2)
    elif kind == "identical rows":
        ts = np.broadcast_to(np.cumsum(rng.normal(100_000, 5_000, size=(B, 1, R)).astype(np.int64), axis=2), (B, n, R))
    elif kind == "equal periods":
        ts = rng.integers(0, 100_000, size=(B, n, 1)) + 100_000 * np.arange(1, R + 1)
    elif kind == "coarse clock":
        ts = np.cumsum(100_000 * np.exp(0.3 * rng.standard_normal((B, n, 1))) * (1 + 0.05 * rng.standard_normal((B, n, R))), axis=2) // 50_000 * 50_000
    elif kind == "small numbers":
        ts = np.cumsum(rng.integers(0, 3, size=(B, n, R)), axis=2)
    elif kind == "power law":
        ts = np.cumsum(1000 * np.minimum((1 - rng.random((B, n, R))) ** (-1 / 1.2), 1e6), axis=2)
    elif kind == "bursts":
        ts = np.cumsum(np.where(rng.random((B, n, R)) < 0.02, rng.random((B, n, R)) * 1e7, rng.random((B, n, R)) * 50), axis=2)
    return np.ascontiguousarray(ts).astype(np.int64)


def check(ts, objective, sel):
    for b in range(min(len(ts), 6)):
        w, t, idx = o.sweep_window(ts[b], objective)
        assert int(sel.status[b]) == 0 and (int(sel.wait[b]), int(sel.barrier[b])) == (w, t), b
        assert (sel.idx[b].cpu().numpy() == idx).all(), b


def us(call, calls=5, groups=5):
    """Fastest of a few groups of calls, microseconds a call."""
    best = float("inf")
    for _ in range(groups):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(calls):
            call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / calls * 1e3)
    return best


def compare(ts, objective, slack):
    """Results of a handle that has settled on its route against the oracle; its time against the other routes'."""
    B, n, R = ts.shape
    d = torch.from_numpy(ts).cuda()
    time = []
    for plain in (True, False):
        h = zl.ZipLine(n, R, B, objective)
        if plain:
            h.set_option("no_cells", 1)
            h.set_option("no_walk", 1)
        sel = h.select_batched(d)
        for _ in range(30):
            h.select_batched(d, sel)
        check(ts, objective, sel)
        time.append(us(lambda: h.select_batched(d, sel)))
        h.destroy()
    assert time[1] <= slack * time[0] + 10, time


@pytest.mark.parametrize("objective", [0, 1])
@pytest.mark.parametrize("n,R,B", [(64, 128, 4), (300, 1024, 4), (93, 211, 64)])
def test_rows_that_stand_still(n, R, B, objective):
    compare(rows("standing still", n, R, B), objective, 2.0)


@pytest.mark.parametrize("kind", ["identical rows", "equal periods", "coarse clock", "small numbers"])
@pytest.mark.parametrize("objective", [0, 1])
@pytest.mark.parametrize("n,R,B", [(64, 128, 4), (100, 150, 1), (93, 211, 64), (128, 256, 100)])
def test_many_selections_of_the_least_wait(n, R, B, objective, kind):
    # the handle leaves the route, or the ties are sorted out
    compare(rows(kind, n, R, B), objective, 1.5)


@pytest.mark.parametrize("kind", ["power law", "bursts", "standing still for long"])
@pytest.mark.parametrize("n,R,B", [(300, 1023, 3), (1024, 1024, 8)])
def test_rows_far_from_arithmetic(n, R, B, kind):
    compare(rows(kind, n, R, B), 0, 2.0)


@pytest.mark.parametrize("kind", ["identical rows", "equal periods", "coarse clock", "small numbers", "wide"])
@pytest.mark.parametrize("n,R,B", [(16, 64, 1500), (16, 64, 2), (33, 24, 700)])
def test_small_instances_with_many_selections_of_the_least_wait(n, R, B, kind):
    ts = rows("coarse clock", n, R, B) * 50_000 if kind == "wide" else rows(kind, n, R, B)
    compare(ts, 0, 1.5)


def test_regular_small_instances_stay_with_a_warp_each():
    import zl_inputs as zi
    for recipe in ("c2", "c3", "c4"):
        for n, R in ((16, 64), (32, 32), (20, 100)):
            ts = torch.from_numpy(zi.generate(zi.CONFIGS[recipe].with_(B=4096, n=n, R=R))).cuda()
            h = zl.ZipLine(n, R, 4096, 0)
            for _ in range(3):
                h.select_batched(ts)
                torch.cuda.synchronize()
            assert h.launches_per_call == 1                        # (4 on the bucket route)
            h.destroy()


def test_small_instances_without_a_handle():
    # no state to learn from: at most twice what a CTA an instance takes, whatever the rows hold
    for n, R, B in ((16, 64, 2), (16, 16, 2), (32, 32, 8)):
        for kind in ("equal periods", "identical rows", "coarse clock"):
            ts = torch.from_numpy(rows(kind, n, R, B)).cuda()
            out = zl.Selection(torch.empty((B, n), dtype=torch.int32, device="cuda"),
                               *(torch.empty(B, dtype=t, device="cuda") for t in (torch.int64, torch.int64, torch.int32)))
            zl.zl_select_batched_noalloc(ts, out, 0)
            check(ts.cpu().numpy(), 0, out)
            h = zl.ZipLine(n, R, B, 0)
            h.set_option("no_cells", 1)
            h.set_option("no_walk", 1)
            sel = h.select_batched(ts)
            plain = us(lambda: h.select_batched(ts, sel))
            t = us(lambda: zl.zl_select_batched_noalloc(ts, out, 0))
            assert t <= 2 * plain + 30, (n, R, kind, t, plain)
            h.destroy()
