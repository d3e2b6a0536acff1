"""The cell route (branch and bound over time cells) against the CPU oracle at the sizes where it can go wrong.  Whole numbers:
every comparison is exact."""
import numpy as np
import pytest
import torch

import oracle as o
import zl_inputs as zi

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2001_01347_b200 as zl


def select(ts, objective, flags=0):
    B, n, R = ts.shape
    h = zl.ZipLine(n, R, B, objective, 0, flags)
    h.set_option("cells", 1)
    assert h.launches_per_call == 2
    sel = h.select_batched(torch.from_numpy(np.ascontiguousarray(ts)).cuda())
    torch.cuda.synchronize()
    left = h.filter_counts(B)[2]
    h.destroy()
    return sel, left


def assert_oracle(ts, objective, sel):
    for b in range(ts.shape[0]):
        w, t, idx = o.sweep_window(ts[b], objective)
        assert int(sel.status[b]) == 0
        assert (int(sel.wait[b]), int(sel.barrier[b])) == (w, t), b
        assert (sel.idx[b].cpu().numpy() == idx).all(), b


@pytest.mark.parametrize("objective", [0, 1])
@pytest.mark.parametrize("n,R,B", [(8, 513, 3), (8, 5000, 2), (15, 300, 5), (17, 257, 160), (31, 133, 9), (33, 129, 2), (63, 67, 700),
                                   (97, 211, 40), (128, 33, 20), (255, 65, 1), (257, 64, 7), (1000, 15, 1), (1025, 9, 3), (4096, 2, 2),
                                   (4095, 130, 1), (10, 150, 3), (64, 64, 700), (300, 13, 600), (129, 8, 2)])
def test_shapes_around_the_pieces_slices_and_clusters(n, R, B, objective):
    # rows of odd length and start (pieces of eight elements on 32-byte boundaries), row counts around the CTAs of a
    # cluster, batches that change its size; spread workers with rare long iterations, so that estimates are off
    w = zi.CONFIGS["c4"].with_(B=B, n=n, R=R)
    ts = zi.generate(w, first_instance=n)
    sel, left = select(ts, objective)
    assert max(left) == 0 or n < 16
    assert_oracle(ts, objective, sel)


@pytest.mark.parametrize("n,R,B", [(4, 1025, 40), (5, 2000, 3), (7, 1218, 34)])
def test_a_handful_of_workers(n, R, B):
    ts = zi.generate(zi.CONFIGS["c4"].with_(B=B, n=n, R=R))
    assert_oracle(ts, 0, select(ts, 0)[0])


@pytest.mark.parametrize("objective", [0, 1])
def test_ties_flat_rows_and_far_from_arithmetic(objective):
    rng = np.random.default_rng(5 + objective)
    for n, R, B, hi in ((40, 120, 6, 3), (100, 60, 4, 2), (300, 30, 3, 40)):
        ts = (rng.integers(0, 5, size=(B, n, 1)) + np.cumsum(rng.integers(0, hi, size=(B, n, R)), axis=2)).astype(np.int64)
        assert_oracle(ts, objective, select(ts, objective)[0])
    inc = np.where(rng.random((9, 64, 100)) < 0.02, 5000, rng.integers(1, 30, size=(9, 64, 100)))
    assert_oracle(np.cumsum(inc, axis=2), objective, select(np.cumsum(inc, axis=2).astype(np.int64), objective)[0])
    ts = np.full((2, 70, 60), 77, dtype=np.int64)                  # one timestamp everywhere
    assert_oracle(ts, objective, select(ts, objective)[0])


@pytest.mark.parametrize("objective", [0, 1])
def test_what_the_cells_leave_over_and_errors(objective):
    # one batch: a regular instance, one whose span needs 64 bits (segment sweep), identical rows, an unsorted one, a
    # negative timestamp
    n, R = 64, 128
    regular = zi.generate(zi.CONFIGS["c3"].with_(B=1, n=n, R=R))[0]
    same = np.broadcast_to(np.cumsum(np.arange(1, R + 1)) * 1000, (n, R))
    unsorted = regular.copy()
    unsorted[5, 60] = unsorted[5, 58] - 1
    negative = regular.copy()
    negative[3, 0] = -4
    ts = np.stack([regular, regular * 50_000, same, unsorted, negative, regular + 9]).astype(np.int64)
    sel, left = select(ts, objective, zl.ZL_FLAG_CHECK_SORTED)
    bad = [0, 0, 0, zl.binding.ZL_ERR_UNSORTED, zl.binding.ZL_ERR_INVALID_ARG, 0]
    assert sel.status.tolist() == bad
    assert (sel.idx[3:5] == -1).all() and (sel.wait[3:5] == np.iinfo(np.int64).min).all()
    keep = [0, 1, 2, 5]
    assert_oracle(ts[keep], objective, zl.Selection(sel.idx[keep], sel.barrier[keep], sel.wait[keep], sel.status[keep]))


@pytest.mark.parametrize("objective", [0, 1])
def test_predicted_rows(objective):
    rng = np.random.default_rng(11)
    for n, R, B in ((16, 300, 5), (100, 150, 3), (513, 200, 2)):
        iv = np.maximum(1, (100_000 * np.exp(0.5 * rng.standard_normal((B, n)))).astype(np.int64))
        last = rng.integers(0, 100_000, size=(B, n))
        h = zl.ZipLine(n, R, B, objective, 0, zl.ZL_FLAG_PREDICTOR)
        h.set_option("cells", 1)
        sel = h.predict_select_batched(torch.from_numpy(last).cuda(), torch.from_numpy(iv).cuda())
        torch.cuda.synchronize()
        assert_oracle(np.stack([o.predict(last[b], iv[b], R) for b in range(B)]), objective, sel)
        h.destroy()


def periodic(n, R, B, seed=3):
    """Workers that all take exactly as long: every period holds a selection of nearly the least wait, far more cells than there
    is room for are left, and the instance goes to the segment sweep."""
    rng = np.random.default_rng(seed)
    return (rng.integers(0, 100_000, size=(B, n, 1)) + 100_000 * np.arange(1, R + 1)).astype(np.int64)


@pytest.mark.parametrize("bad_rows", ["periodic", "wide"])
@pytest.mark.parametrize("objective", [0, 1])
def test_a_handle_takes_the_route_after_its_first_calls_and_leaves_it_when_it_fails(objective, bad_rows):
    n, R, B = 64, 512, 4
    ts = zi.generate(zi.CONFIGS["c3"].with_(B=B, n=n, R=R))
    rows = periodic(n, R, B) if bad_rows == "periodic" else ts * 50_000           # lists that overflow; spans beyond 32 bits
    good, bad = torch.from_numpy(ts).cuda(), torch.from_numpy(rows).cuda()
    if bad_rows == "periodic":
        assert max(select(rows, objective)[1]) == 1
    h = zl.ZipLine(n, R, B, objective)

    def calls(k, on_cells):
        for _ in range(k):
            assert (h.launches_per_call == 2) == on_cells
            assert_oracle(ts, objective, h.select_batched(good))
    calls(8, False)
    for _ in range(2):                                             # the second failure waits as long as the first: it was made good
        calls(3, True)
        for _ in range(10):                                        # several are under way when the first one's word arrives
            sel = h.select_batched(bad)
        assert_oracle(rows, objective, sel)
        torch.cuda.synchronize()
        assert h.launches_per_call != 2
        while h.launches_per_call != 2:
            h.select_batched(good)
        calls(1, True)
        torch.cuda.synchronize()
        calls(40, True)                                            # the late words are not booked against the new run of calls
    h.select_batched(bad)
    torch.cuda.synchronize()
    calls(17, False)                                               # the call that sees the word, then the 16 of a first failure
    calls(1, True)
    h.select_batched(bad)                                          # a second failure in a row waits twice as long
    torch.cuda.synchronize()
    calls(33, False)
    calls(1, True)
    h.destroy()


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("wide", [False, True])
def test_host_rows_read_in_place_or_copied(pinned, wide):
    # just above 2^18 timestamps; a batch with an instance that the cells leave over is copied after all, one with an instance in
    # error is not
    n, R, B = 65, 257, 16
    ts = zi.generate(zi.CONFIGS["c4"].with_(B=B, n=n, R=R))
    if wide:
        ts[3] *= 50_000
    t = torch.from_numpy(ts).pin_memory() if pinned else torch.from_numpy(ts)
    h = zl.ZipLine(n, R, B, 0)
    before = h.workspace_bytes
    for _ in range(2):
        assert_oracle(ts, 0, h.select_batched_host(t))
    t[5, 0, 0] = -1
    for _ in range(2):
        sel = h.select_batched_host(t)
        keep = [b for b in range(B) if b != 5]
        assert sel.status[5] == zl.binding.ZL_ERR_INVALID_ARG and (sel.idx[5] == -1).all() and sel.wait[5] == np.iinfo(np.int64).min
        assert_oracle(ts[keep], 0, zl.Selection(sel.idx[keep], sel.barrier[keep], sel.wait[keep], sel.status[keep]))
    assert (h.workspace_bytes - before >= ts.nbytes) == (wide or not pinned)       # the staging buffer of the copy
    h.destroy()


@pytest.mark.parametrize("n,R,B", [(1, 1, 3), (1, 64, 2), (4, 64, 3), (32, 8, 5), (33, 7, 4), (64, 4, 3), (65, 3, 3), (128, 2, 3), (128, 4, 700),
                                   (16, 31, 601), (16, 64, 2500), (31, 33, 2400), (5, 100, 3), (32, 32, 5), (65, 47, 1300), (128, 24, 1200), (20, 100, 1201)])
@pytest.mark.parametrize("values", ["spread", "ties", "wide"])
def test_small_instances_a_warp_each(n, R, B, values):
    # one to four rows a lane, the last row of a lane missing, one warp a CTA and four, the last CTA not full
    rng = np.random.default_rng(n * 1000 + R)
    hi = {"spread": 10 ** 6, "ties": 3, "wide": 10 ** 9}[values]
    ts = (rng.integers(0, 3 * hi, size=(B, n, 1)) + np.cumsum(rng.integers(0, hi, size=(B, n, R)), axis=2)).astype(np.int64)
    if B > 3 and R > 2:
        ts[1, n // 2, 1] = ts[1, n // 2, 0] - 1                    # not sorted
        ts[3, 0, 0] = -1
    h = zl.ZipLine(n, R, B, 0, 0, zl.ZL_FLAG_CHECK_SORTED)
    assert h.launches_per_call == 1
    sel = h.select_batched(torch.from_numpy(ts).cuda())
    torch.cuda.synchronize()
    status, wait, barrier, idx = (x.cpu().numpy() for x in (sel.status, sel.wait, sel.barrier, sel.idx))
    for b in range(min(B, 200)):
        if B > 3 and R > 2 and b in (1, 3):
            assert status[b] in (zl.binding.ZL_ERR_UNSORTED, zl.binding.ZL_ERR_INVALID_ARG) and (idx[b] == -1).all()
            continue
        w, t, ix = o.sweep_window(ts[b], 0)
        assert status[b] == 0 and (int(wait[b]), int(barrier[b])) == (w, t) and (idx[b] == ix).all(), b
    h.set_option("no_walk", 1)                                     # the rest of the batch: a CTA an instance
    ref = h.select_batched(torch.from_numpy(ts).cuda())
    assert torch.equal(ref.idx, sel.idx) and torch.equal(ref.wait, sel.wait) and torch.equal(ref.barrier, sel.barrier) and torch.equal(ref.status, sel.status)
    h.destroy()


@pytest.mark.parametrize("n,R,B", [(4, 8, 3), (16, 64, 700), (33, 20, 700), (100, 10, 3)])
def test_small_instances_with_a_time_before_every_first_element(n, R, B):
    # rows that are not sorted, and not checked to be: what an instance's result is is not defined, but it stays within its own
    # buffers, and the others are right
    rng = np.random.default_rng(n)
    ts = (1000 + np.cumsum(rng.integers(1, 10 ** 6, size=(B, n, R)), axis=2)).astype(np.int64)
    broken = ts.copy()
    for back in (1, 2, 1 << 20):
        broken[1] = ts[1]
        broken[1, n - 1, 1:-1] = ts[1, :, 0].min() - back
        h = zl.ZipLine(n, R, B, 0)
        assert h.launches_per_call == 1
        sel = h.select_batched(torch.from_numpy(broken).cuda())
        torch.cuda.synchronize()
        keep = [0] + list(range(2, min(B, 60)))
        assert_oracle(ts[keep], 0, zl.Selection(sel.idx[keep], sel.barrier[keep], sel.wait[keep], sel.status[keep]))
        h.destroy()


def test_host_rows_in_two_pinned_regions_are_not_read_in_place():
    # the first and the last pages are registered, what lies between is not: the rows are copied (or the copy is refused), and the
    # staging buffer of the copy exists afterwards
    import mmap
    n, R, B = 65, 257, 16
    ts = zi.generate(zi.CONFIGS["c4"].with_(B=B, n=n, R=R))
    page, size = mmap.PAGESIZE, ts.nbytes
    total = -(-size // page) * page
    m = mmap.mmap(-1, total)
    a = np.frombuffer(m, dtype=np.int64, count=ts.size).reshape(ts.shape)
    a[...] = ts
    t = torch.from_numpy(a)
    rt = torch.cuda.cudart()
    ends = ((t.data_ptr(), 4 * page), (t.data_ptr() + total - 4 * page, 4 * page))
    for p, k in ends:
        assert int(rt.cudaHostRegister(p, k, 0)) == 0
    h = zl.ZipLine(n, R, B, 0)
    before = h.workspace_bytes
    try:
        assert_oracle(ts, 0, h.select_batched_host(t))
    except zl.ZipLineError as e:
        assert e.code == zl.binding.ZL_ERR_CUDA
    finally:
        assert h.workspace_bytes - before >= size
        assert_oracle(ts, 0, h.select_batched(torch.from_numpy(ts).cuda()))    # (a refused copy is not reported once more)
        h.destroy()
        for p, _ in ends:
            assert int(rt.cudaHostUnregister(p)) == 0


@pytest.mark.parametrize("objective", [0, 1])
@pytest.mark.parametrize("short", [0, 16, 999, 1 << 18, (1 << 20) + 7])
@pytest.mark.parametrize("n,R", [(64, 128), (300, 40), (20, 300)])
def test_the_last_cell_of_a_timeline_that_ends_just_below_32_bits(n, R, short, objective):
    # every row ends at the same time, up to the largest that 32 bits hold: the optimum (0) is the last element, in the cell
    # that 2^32 cuts.  One row has an element shortly before, so that no cell before it sees the last one as its first.
    end = (1 << 32) - 4 - short
    rng = np.random.default_rng(n + short)
    inner = np.sort(rng.integers(1, end - (1 << 21), size=(3, n, R - 2)), axis=2)
    first, last = np.arange(3 * n).reshape(3, n, 1) % 7, np.full((3, n, 1), end)
    first[:, 0] = 0
    ts = np.concatenate([first, inner, last], axis=2).astype(np.int64)
    ts[:, 1, R - 2] = end - (6 << 16)
    assert (np.diff(ts, axis=2) >= 0).all()
    assert_oracle(ts, objective, select(ts, objective)[0])
    ts += 12_345
    d = torch.from_numpy(ts).cuda()
    out = zl.Selection(torch.empty((3, n), dtype=torch.int32, device="cuda"), *(torch.empty(3, dtype=t, device="cuda") for t in (torch.int64, torch.int64, torch.int32)))
    zl.zl_select_batched_noalloc(d, out, objective)
    torch.cuda.synchronize()
    assert_oracle(ts, objective, out)


@pytest.mark.parametrize("objective,n,R,few,many", [(0, 64, 48, 2, 1), (0, 128, 20, 2, 1), (0, 300, 12, 5, 2), (1, 300, 12, 5, 2)])
def test_the_route_follows_the_instances_of_the_call(objective, n, R, few, many):
    # one instance on a handle with room for 4096: the kernels that are best for one (the bucket route's, or the cells where
    # they are), not those that are best for 4096
    ts = zi.generate(zi.CONFIGS["c3"].with_(B=1300, n=n, R=R))
    d = torch.from_numpy(ts).cuda()
    h = zl.ZipLine(n, R, 4096, objective)
    for _ in range(10):
        one = h.select_batched(d[:1].contiguous())
    assert h.launches_per_call == few
    assert_oracle(ts[:1], objective, one)
    for _ in range(10):
        sel = h.select_batched(d)
    assert h.launches_per_call == many
    assert_oracle(ts[:40], objective, zl.Selection(sel.idx[:40], sel.barrier[:40], sel.wait[:40], sel.status[:40]))
    one = h.select_batched(d[:1].contiguous())
    assert h.launches_per_call == few
    assert torch.equal(one.idx[0], sel.idx[0]) and one.wait[0] == sel.wait[0]
    h.destroy()
