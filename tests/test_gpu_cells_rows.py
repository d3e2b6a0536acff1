"""The cell route's ways of reading rows and of passing answers on, at the sizes where they can go wrong, against the CPU oracle.
Whole numbers: every comparison is exact."""
import numpy as np
import pytest
import torch

import oracle as o
import zl_inputs as zi

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2001_01347_b200 as zl


def check(ts, objective, offset=0, instances=None, leaves=0):
    """The cell route, and nothing else, on rows that start `offset` timestamps behind a 32-byte boundary; `leaves`: instances that may be
    left to the segment sweep.  (What lies outside the matrix is mapped here; tests/test_cells_rows_on_cpu.py looks at every load.)"""
    B, n, R = ts.shape
    flat = torch.empty(offset + ts.size, dtype=torch.int64, device="cuda")
    d = flat[offset:].view(B, n, R)
    d.copy_(torch.from_numpy(ts))
    h = zl.ZipLine(n, R, B, objective, 0)
    h.set_option("cells", 1)
    h.set_option("no_walk", 1)
    sel = h.select_batched(d)
    torch.cuda.synchronize()
    assert h.launches_per_call == 2
    assert sum(x != 0 for x in h.filter_counts(B)[2]) <= leaves
    for b in range(B) if instances is None else instances:
        w, t, idx = o.sweep_window(ts[b], objective)
        assert (int(sel.status[b]), int(sel.wait[b]), int(sel.barrier[b])) == (0, w, t), b
        assert (sel.idx[b].cpu().numpy() == idx).all(), b
    h.destroy()


@pytest.mark.parametrize("objective", [0, 1])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
@pytest.mark.parametrize("n,R,B", [(4, 1, 1), (4, 2, 1), (5, 3, 2), (7, 9, 1), (8, 8, 3), (33, 31, 2), (100, 150, 1)])
def test_pieces_at_the_ends_of_the_matrix(n, R, B, offset, objective):
    # eight elements on a 32-byte boundary may begin before the first row or end behind the last one
    check(zi.generate(zi.CONFIGS["c4"].with_(B=B, n=n, R=R)), objective, offset)


@pytest.mark.parametrize("objective", [0, 1])
@pytest.mark.parametrize("n,R,B", [(1023, 40, 2), (1024, 40, 2), (1025, 40, 2), (2049, 33, 1), (1024, 8200, 1), (300, 14000, 8), (200, 100, 400), (64, 12, 1000), (300, 12, 1000)])
def test_lists_of_rows_and_shapes_of_clusters(n, R, B, objective):
    # one list of 1024 rows and more than one, counts of pieces beyond 20 bits, clusters of 16 and 10, three CTAs an SM, many of short rows
    check(zi.generate(zi.CONFIGS["c4"].with_(B=B, n=n, R=R)), objective, 1, range(0, B, max(1, B // 3)))


@pytest.mark.parametrize("objective", [0, 1])
@pytest.mark.parametrize("share", [0.02, 0.2])
def test_rows_far_off_their_estimates(share, objective):
    # bursts: rows are read on to either side of what was estimated, one cell holds many elements of a row
    rng = np.random.default_rng(3)
    inc = np.where(rng.random((3, 200, 600)) < share, rng.integers(1, 100_000, (3, 200, 600)), rng.integers(1, 50, (3, 200, 600)))
    # (SUM, the smaller share: two of the instances keep more cells than there is room for)
    check(np.cumsum(inc, axis=2).astype(np.int64), objective, leaves=2 if objective == 1 and share == 0.02 else 0)


@pytest.mark.parametrize("objective", [0, 1])
@pytest.mark.parametrize("fast", [1, 20, 45])
def test_fast_workers_in_one_cta(fast, objective):
    # the first CTA of the cluster has the fast workers; SUM: more than the 32 answers that a warp evaluates by itself
    rng = np.random.default_rng(fast)
    m = np.where(np.arange(160) < fast, 1000, 100_000)[None, :, None]
    check(np.cumsum((m * (1 + 0.05 * rng.standard_normal((2, 160, 400)))).astype(np.int64), axis=2), objective)


@pytest.mark.parametrize("seed", [0, 1, 3])
def test_more_answers_from_one_cta_than_its_share_sum(seed):
    # bursts: one run of cells holds dozens of elements of a row (one to four exchanges an instance fetch answers from where they were put)
    rng = np.random.default_rng(seed)
    inc = np.where(rng.random((3, 200, 600)) < 0.03, rng.integers(1, 100_000, (3, 200, 600)), rng.integers(1, 50, (3, 200, 600)))
    check(np.cumsum(inc, axis=2).astype(np.int64), 1)


@pytest.mark.parametrize("jitter", [0, 0.0005])
def test_more_answers_from_one_cta_than_its_share_range(jitter):
    # the first CTA has the slow workers, all of one period and close together: forty answers to each of several runs of cells
    rng = np.random.default_rng(1)
    m = np.where(np.arange(320) < 40, 100_000, 3000)[None, :, None]
    check(np.cumsum((m * (1 + jitter * rng.standard_normal((2, 320, 200)))).astype(np.int64), axis=2) + rng.integers(0, 1000, (2, 320, 1)), 0)


@pytest.mark.parametrize("objective", [0, 1])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
@pytest.mark.parametrize("n,R,B", [(4, 2, 1), (7, 9, 2), (24, 60, 1), (128, 20, 100), (90, 60, 700), (1088, 64, 64), (1088, 128, 32), (1280, 32, 64), (300, 400, 2)])
def test_every_load_of_the_rows_is_inside_them(n, R, B, offset, objective):
    ts = zi.generate(zi.CONFIGS["c1"].with_(B=B, n=n, R=R))
    d = torch.empty(offset + ts.size, dtype=torch.int64, device="cuda")[offset:].view(ts.shape)
    d.copy_(torch.from_numpy(ts))
    h = zl.ZipLine(n, R, B, objective, 0, zl.ZL_FLAG_DEBUG_CHECKS)
    h.set_option("cells", 1)
    h.set_option("no_walk", 1)
    sel = h.select_batched(d)
    torch.cuda.synchronize()
    assert h.launches_per_call == 2 and max(h.filter_counts(B)[2]) == 0
    assert h.debug_report() == (0, 0, 0)
    assert h.check_canaries()[1] == 0
    for b in (0, B - 1):
        w, t, idx = o.sweep_window(ts[b], objective)
        assert (int(sel.status[b]), int(sel.wait[b]), int(sel.barrier[b])) == (0, w, t), b
        assert (sel.idx[b].cpu().numpy() == idx).all(), b
    h.destroy()


def on(route, ts, n, R, B, objective):
    h = zl.ZipLine(n, R, B, objective, 0)
    for option in route:
        h.set_option(option, 1)
    sel = h.select_batched(ts)
    torch.cuda.synchronize()
    launches, left = h.launches_per_call, h.filter_counts(B)[2]
    h.destroy()
    return sel, launches, left


@pytest.mark.parametrize("R", [7, 8, 9, 63, 64])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_a_decrease_is_reported_wherever_it_is(R, offset):
    # an instance for every place of the decrease, and one without
    n = 9 if R < 63 else 5
    places = [f for f in range(n * R) if f % R]
    ts = np.tile(1000 + 2 * np.arange(1, R + 1), (len(places) + 1, n, 1)).astype(np.int64)
    flat = ts.reshape(len(places) + 1, n * R)
    for b, f in enumerate(places):
        flat[b, f] = flat[b, f - 1] - 1
    d = torch.empty(offset + ts.size, dtype=torch.int64, device="cuda")[offset:].view(ts.shape)
    d.copy_(torch.from_numpy(ts))
    for objective in (0, 1):
        h = zl.ZipLine(n, R, len(ts), objective, 0, zl.ZL_FLAG_CHECK_SORTED)
        h.set_option("cells", 1)
        h.set_option("no_walk", 1)
        sel = h.select_batched(d)
        torch.cuda.synchronize()
        assert h.launches_per_call == 2
        assert sel.status.tolist() == [zl.binding.ZL_ERR_UNSORTED] * len(places) + [0], objective
        h.destroy()


@pytest.mark.parametrize("recipe", ["c3", "c4"])
@pytest.mark.parametrize("n,R,B", [(90, 60, 400), (40, 30, 500), (90, 60, 500), (90, 60, 700), (90, 60, 900), (90, 60, 1000), (120, 20, 1100),
                                   (511, 12, 1000), (512, 12, 1000), (513, 12, 1000), (600, 25, 1200), (300, 60, 1150), (30, 600, 760)])
def test_every_form_of_ctas_that_share_an_sm(n, R, B, recipe):
    # three to eight CTAs an SM, few and many timestamps for their threads, one list of 512 rows and more than one, few rows
    # with a long lookahead: every instance as the filter or bucket route has it, some as the oracle does
    d = torch.from_numpy(zi.generate(zi.CONFIGS[recipe].with_(B=B, n=n, R=R))).cuda()
    sel, launches, left = on(("cells", "no_walk"), d, n, R, B, 0)
    assert launches == 2 and max(left) == 0
    other, launches, _ = on(("no_cells", "no_walk"), d, n, R, B, 0)
    assert launches != 2
    for a, b in zip((sel.idx, sel.barrier, sel.wait, sel.status), (other.idx, other.barrier, other.wait, other.status)):
        assert torch.equal(a, b)
    for b in range(0, B, B // 4):
        w, t, idx = o.sweep_window(d[b].cpu().numpy(), 0)
        assert (int(sel.wait[b]), int(sel.barrier[b])) == (w, t), b
        assert (sel.idx[b].cpu().numpy() == idx).all(), b


@pytest.mark.parametrize("recipe", ["c3", "c4"])
@pytest.mark.parametrize("n,R,B", [(90, 60, 297), (90, 100, 400), (1024, 16, 300), (1025, 16, 300), (100, 60, 444), (128, 64, 445), (129, 64, 445), (90, 120, 592), (90, 120, 593)])
def test_every_form_of_ctas_that_share_an_sm_sum(n, R, B, recipe):
    # three and four CTAs an SM, the first and last batch of each, few and many timestamps, one list of rows and more than one.  (A form
    # that gave up would leave every instance to the segment sweep; that a few keep too many cells depends on their rows.)
    d = torch.from_numpy(zi.generate(zi.CONFIGS[recipe].with_(B=B, n=n, R=R))).cuda()
    sel, launches, left = on(("cells", "no_walk"), d, n, R, B, 1)
    assert launches == 2 and sum(x != 0 for x in left) < B // 10
    other, launches, _ = on(("no_cells", "no_walk"), d, n, R, B, 1)
    assert launches != 2
    for a, b in zip((sel.idx, sel.barrier, sel.wait, sel.status), (other.idx, other.barrier, other.wait, other.status)):
        assert torch.equal(a, b)
    for b in range(0, B, B // 4):
        w, t, idx = o.sweep_window(d[b].cpu().numpy(), 1)
        assert (int(sel.wait[b]), int(sel.barrier[b])) == (w, t), b
        assert (sel.idx[b].cpu().numpy() == idx).all(), b


def test_what_crowded_ctas_leave_over():
    # workers in step: more answers, or more cells, than a CTA of seven an SM has room for; the segment sweep takes the instances
    n, R, B = 1000, 20, 1000
    rng = np.random.default_rng(4)
    ts = 100_000 * np.arange(1, R + 1) + rng.integers(0, 500, (4, n, R)) + np.where(np.arange(n) < 200, 0, rng.integers(0, 100_000, n))[None, :, None]
    ts = np.sort(ts.astype(np.int64), axis=2)
    sel, launches, left = on(("cells", "no_walk"), torch.from_numpy(ts).cuda().repeat(B // 4, 1, 1), n, R, B, 0)
    assert launches == 2 and max(left) == 1
    for b in (0, 1, 2, 3, B - 1):
        w, t, idx = o.sweep_window(ts[b % 4], 0)
        assert (int(sel.status[b]), int(sel.wait[b]), int(sel.barrier[b])) == (0, w, t), b
        assert (sel.idx[b].cpu().numpy() == idx).all(), b
