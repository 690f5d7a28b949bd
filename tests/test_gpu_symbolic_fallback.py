"""The device symbolic phase where its tables do not hold every row: the retry of
the small table on the large one, rows of A longer than the large one, and a row
that outgrows it only by fill; always the host phase's pattern."""
from __future__ import annotations

import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1703_01325_gb300.bilu as B  # noqa: E402
from paper_1703_01325_gb300 import _lib as L  # noqa: E402

pytestmark = pytest.mark.gpu


def _csr(cols):
    cols = [sorted(c) for c in cols]
    return (np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int32),
            np.concatenate(cols).astype(np.int32))


def _symbolic_launches(n, rp, ci, k, cap):
    """The device pattern, checked against the host's, and how many row kernels it took (the symbolic class)."""
    lib = L.load()
    count, ms = C.c_int64(), C.c_double()
    lib.bilu_profile_enable(1)
    try:
        g = B.bilu_symbolic_gpu(n, rp, ci, k, row_capacity=cap)
        assert lib.bilu_profile_read(L.PROF_KERNELS.index("symbolic"), C.byref(count), C.byref(ms)) == L.BILU_OK
        launches = count.value
    finally:
        lib.bilu_profile_enable(0)
    eg, eh = g.export(), B.bilu_symbolic(n, rp, ci, k).export()
    for key in eh:
        assert np.array_equal(eg[key], eh[key]), key
    return launches


def _tree(levels, degree, reverse):
    """Cells of a tree, numbered from the leaves up (or from the root down: no fill), each tied to its children."""
    sizes = [degree ** q for q in range(levels + 1)]
    n = sum(sizes)
    cols = [{i} for i in range(n)]
    first = np.concatenate([[0], np.cumsum(sizes)])
    for q in range(levels):
        for x in range(sizes[q]):
            for c in range(degree):
                a, b = first[q] + x, first[q + 1] + x * degree + c
                if not reverse:
                    a, b = n - 1 - a, n - 1 - b
                cols[a].add(int(b))
                cols[b].add(int(a))
    return n, *_csr(cols)


def _vertices_met(n, rp, ci, i, k):
    """How many vertices the walks of length up to k + 1 from row i put into its table: walks go on over vertices
    numbered below i, and of the longest ones only fill paths (largest interior vertex below both ends) count."""
    met = {int(v) for v in ci[rp[i]:rp[i + 1]]}
    cur = {v: -1 for v in met if v != i}  # least largest interior vertex of the walks of the current length
    for d in range(1, k + 1):
        nxt = {}
        for u, top in cur.items():
            if u >= i:
                continue
            top = max(top, u)
            for v in ci[rp[u]:rp[u + 1]]:
                v = int(v)
                if v in (i, u) or (d == k and top >= min(i, v)):
                    continue
                met.add(v)
                if v < i:
                    nxt[v] = min(nxt.get(v, n), top)
        cur = nxt
    return len(met)


@pytest.mark.parametrize("k", [2, 3])
def test_small_table_retries_on_the_large_one(libbilu, k):
    """Rows of A of at most 8 entries (the small table, 96 vertices) that meet between 97 and 384: one pass on each
    table, and the rows written from the large one."""
    torch.cuda.set_device(0)
    n, rp, ci = _tree(3, 6, reverse=False)
    assert int(np.diff(rp).max()) <= 8
    most = max(_vertices_met(n, rp, ci, i, k) for i in range(n))
    if k == 3:
        assert 96 < most <= 384
        want = 3  # counted on the small table, on the large one, written
    else:
        assert most <= 96
        want = 2
    assert _symbolic_launches(n, rp, ci, k, 400) == want


@pytest.mark.parametrize("width,cap,want", [(384, 500, 2), (385, 500, 1), (600, 700, 1), (300, 500, 2)])
def test_rows_longer_than_the_table_go_straight_to_the_merges(libbilu, width, cap, want):
    """One row of A of `width` entries without fill: counted and written by paths, or merged at once."""
    torch.cuda.set_device(0)
    cols = [{i} for i in range(3000)]
    cols[1000] |= set(range(1000 - width + 1, 1000))
    assert _symbolic_launches(3000, *_csr(cols), 1, cap) == want


def test_one_row_outgrows_the_table_by_fill(libbilu):
    """Rows of A of 21 entries; the last one meets more than 384 vertices at k = 1: paths on the large table, then
    merges."""
    torch.cuda.set_device(0)
    cols = [{i} for i in range(2000)]
    for c in range(20):
        cols[1500].add(c)
        cols[c] |= set(range(100 + 20 * c, 120 + 20 * c))
    rp, ci = _csr(cols)
    assert _vertices_met(2000, rp, ci, 1500, 1) > 384
    assert _symbolic_launches(2000, rp, ci, 1, 600) == 2
