"""How the cell route reads rows, on the CPU: the device functions are cut out of the kernel's source and run by coroutines (32 to a
warp), every load checked against the matrix.  On a GPU a load behind the end of the matrix nearly always finds other memory."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

import paper_2001_01347_b200.build as build
import zl_inputs as zi

HOST = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host")
RANGE, SUM = 0, 1


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    text = open(os.path.join(build.CSRC, "cells.cu")).read()
    reg = r'"=l"\(([^()]*)\)'
    text = re.sub(r'asm volatile\("ld\.global\.nc\.v4\.u64 [^"]*" : %s : "l"\(([^;]*)\)\);' % ", ".join([reg] * 4), r"load4((uint64_t &)\1, (uint64_t &)\2, (uint64_t &)\3, (uint64_t &)\4, \5);", text)
    text = re.sub(r'asm volatile\("prefetch\.global\.L2 [^"]*"\s*::\s*"l"\(([^;]*)\)\);', r"prefetched(\1);", text)
    rows = text[text.index("template <class SRC> struct RowReader;"): text.index("// ---", text.index("static __device__ bool rows_unsorted"))]
    start = text.rindex("template <", 0, re.search(r"void look_through\(", text).start())
    look = text[start: text.index("\n}\n", start) + 3]
    slack = re.search(r"constexpr int CELL_SLACK = .*", text).group(0)
    assert "asm" not in rows + look
    d = tmp_path_factory.mktemp("rows")
    (d / "rows.inc").write_text(slack + "\n" + rows)
    (d / "look.inc").write_text(look)
    so = str(d / "rows.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-w", '-DROWS_FILE="%s"' % (d / "rows.inc"), '-DLOOK_FILE="%s"' % (d / "look.inc"), "-o", so,
                    os.path.join(HOST, "row_list.cpp")], check=True)
    lib = ctypes.CDLL(so)
    lib.look.restype = lib.places.restype = lib.unsorted.restype = ctypes.c_long
    return lib


def at_offset(ts, offset):
    """The same numbers `offset` timestamps behind a 32-byte boundary."""
    flat = np.empty(ts.size + 8, dtype=np.int64)
    skip = (-(flat.ctypes.data // 8) + offset) % 4
    out = flat[skip: skip + ts.size].reshape(ts.shape)
    out[...] = ts
    return out


def ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


def look(lib, ts, b, objective, a, bnd, shift, slack=4, gap=0, span=0.0, stage=0, threads=128, rows=1024):
    B, n, R = ts.shape
    tmin = int(ts[b].min())
    ends = np.ascontiguousarray((ts[b][:, [0, -1]] - tmin + 1).astype(np.uint32))
    m = ((bnd - 1 - a) >> shift) + 1
    cell, sums, worst = np.zeros((m + 131) & ~3, dtype=np.uint32), np.zeros(2, dtype=np.uint64), np.zeros(1, dtype=np.int64)
    u = ctypes.c_uint32
    bad = lib.look(objective, rows, ptr(ts), B, n, R, b, ctypes.c_int64(tmin), ptr(ends), u(a), u(bnd), u(shift), u(m), u(gap), ctypes.c_float(span), slack, stage, threads,
                   ptr(cell), ptr(sums), ptr(worst))
    assert bad == 0, f"{bad} loads from outside the matrix, up to {worst[0]} timestamps"
    return cell[:m].astype(np.int64), [int(x) for x in sums]


def check_slice(lib, ts, b, objective, a, bnd, shift, slack, threads, rows=1024):
    """Cells and sums of the slice against the rows themselves."""
    T = ts[b].astype(np.int64) - int(ts[b].min()) + 1
    cell, sums = look(lib, ts, b, objective, a, bnd, shift, slack, threads=threads, rows=rows)
    start = a + (np.arange(len(cell), dtype=np.int64) << shift)
    if objective == SUM:
        want = np.zeros(len(cell), dtype=np.int64)
        inside = (T >= a) & (T < bnd)
        np.add.at(want, ((T - a) >> shift)[inside], np.diff(T, axis=1, prepend=0)[inside])
        assert (cell == want).all() and sums[1] == want.sum()
        before = (T < a).sum(axis=1)
        assert sums[0] == sum(int(T[p, k - 1]) for p, k in enumerate(before) if k)
    else:
        inf = 0xffffffff
        G = np.full(len(cell), T[:, 0].max())
        for row in T:
            k = np.searchsorted(row, start)
            G = np.maximum(G, np.where(k < len(row), row[np.minimum(k, len(row) - 1)], inf))
        assert (np.maximum(np.maximum.accumulate(cell), T[:, 0].max()) == G).all()


def slices(T, objective, parts):
    """The route's range of an instance, cut into `parts` CTAs' slices of cells."""
    lo, hi = (1, T[:, -1].min() + 1) if objective == RANGE else (T[:, 0].max(), max(T[:, 0].max(), T[:, -1].min()) + 1)
    lo, hi = int(lo), int(hi)
    shift = max(0, int((hi - lo) / 2000).bit_length() - 1)
    cells = ((hi - lo - 1) >> shift) + 1
    per = ((cells + parts - 1) // parts + 3) & ~3
    for c0 in range(0, cells, per):
        c1 = min(c0 + per, cells)
        yield lo + (c0 << shift), hi if c1 == cells else lo + (c1 << shift), shift


# few and many pieces to a warp, rows shorter than a piece, batches of rows with a few left over, and matrices that end with a page
SHAPES = [(24, 60, 1, 1), (4, 2, 1, 1), (7, 9, 2, 1), (100, 150, 1, 8), (128, 20, 3, 1), (93, 211, 2, 1), (1088, 64, 2, 2), (1088, 128, 1, 2), (1280, 32, 2, 2), (1025, 40, 1, 4)]


@pytest.mark.parametrize("objective", [RANGE, SUM])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
@pytest.mark.parametrize("n,R,B,parts", SHAPES)
def test_every_load_is_inside_the_matrix(lib, n, R, B, parts, offset, objective):
    ts = at_offset(zi.generate(zi.CONFIGS["c1"].with_(B=B, n=n, R=R)), offset)
    b = B - 1                                   # behind the last instance there is nothing
    T = ts[b] - ts[b].min() + 1
    for i, (a, bnd, shift) in enumerate(slices(T, objective, parts)):
        check_slice(lib, ts, b, objective, a, bnd, shift, 4, 128 if i % 2 else 256, (1024, 256, 512)[i % 3])


@pytest.mark.parametrize("objective", [RANGE, SUM])
@pytest.mark.parametrize("share", [0.02, 0.2])
def test_rows_far_off_their_estimates(lib, share, objective):
    # bursts: what the estimate misses is read on to either side
    rng = np.random.default_rng(3)
    inc = np.where(rng.random((2, 60, 300)) < share, rng.integers(1, 100_000, (2, 60, 300)), rng.integers(1, 50, (2, 60, 300)))
    ts = at_offset(np.cumsum(inc, axis=2).astype(np.int64), 1)
    for a, bnd, shift in slices(ts[1] - ts[1].min() + 1, objective, 4):
        check_slice(lib, ts, 1, objective, a, bnd, shift, 4, 128)


def test_a_row_is_searched_inside_the_matrix(lib):
    rng = np.random.default_rng(5)
    for n, R, offset, share in ((3, 1, 1, 0.5), (5, 2, 3, 0.5), (9, 7, 2, 0.5), (20, 64, 0, 0.1), (20, 301, 3, 0.02)):
        inc = np.where(rng.random((2, n, R)) < share, rng.integers(1, 100_000, (2, n, R)), rng.integers(0, 50, (2, n, R)))
        ts = at_offset(np.cumsum(inc, axis=2).astype(np.int64), offset)
        for b in (0, 1):
            tmin = int(ts[b].min())
            T = ts[b] - tmin + 1
            row = np.repeat(np.arange(n, dtype=np.int32), 3 * R)
            t = (T[:, :, None] + np.array([-1, 0, 1])).reshape(-1).astype(np.uint32)
            at, worst = np.zeros(row.size, dtype=np.int32), np.zeros(1, dtype=np.int64)
            bad = lib.places(ptr(ts), 2, n, R, b, ctypes.c_int64(tmin), ptr(np.ascontiguousarray(T[:, [0, -1]].astype(np.uint32))), row.size, ptr(row), ptr(t), ptr(at), ptr(worst))
            assert bad == 0, worst
            assert all(at[i] == np.searchsorted(T[row[i]], t[i]) for i in range(row.size))


@pytest.mark.parametrize("R", [1, 7, 8, 9, 63, 64])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_a_decrease_is_seen_wherever_it_is(lib, R, offset):
    rows = 1100 // R + 1
    ts = at_offset(np.cumsum(np.ones((rows, R), dtype=np.int64), axis=1), offset)
    flat = ts.reshape(-1)
    any_, worst = np.zeros(1, dtype=np.int32), np.zeros(1, dtype=np.int64)

    def seen():
        assert lib.unsorted(ptr(ts), rows, R, 64, ptr(any_), ptr(worst)) == 0, worst
        return bool(any_[0])
    assert not seen()
    for f in range(flat.size):
        if f % R == 0:
            continue
        if R > 9 and f % 61 and (f + offset) % 512 not in (0, 1, 511):
            continue                            # long rows: a sample, and the borders of what a warp takes at once
        flat[f] -= 2
        assert seen(), f
        flat[f] += 2
