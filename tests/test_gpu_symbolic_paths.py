"""The device symbolic phase by fill paths against the host phase, entry for
entry (P', levels of fill, Eq. 4 levels) and through the backfill map (the
factors of one matrix on both patterns, bit for bit): every k up to the merges'
range, rows on both sides of the short-row table, rows that outgrow the large
table and fall back to the merges, the row capacity at its limit, malformed
patterns, row counts around the runs of 32 rows of the level pass."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1703_01325_gb300.reservoir import grid_pattern, random_pattern  # noqa: E402
from tests.oracle_helpers import diag_dominant_block_values  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B(libbilu):
    import paper_1703_01325_gb300.bilu as B
    torch.cuda.set_device(0)
    return B


def _same(B, n, rp, ci, k, cap=1024):
    g, h = B.bilu_symbolic_gpu(n, rp, ci, k, row_capacity=cap), B.bilu_symbolic(n, rp, ci, k)
    eg, eh = g.export(), h.export()
    for key in eh:
        assert np.array_equal(eg[key], eh[key]), key
    for f in ("nnz_p", "nnz_l", "nnz_u", "nlev_l", "nlev_u"):
        assert getattr(g.info, f) == getattr(h.info, f), f
    vals = torch.from_numpy(diag_dominant_block_values(n, 2, rp, ci, 3).reshape(-1)).cuda()
    Fg, Fh = (B.bilu_factor(P.upload(), 2, vals)[0] for P in (g, h))
    assert torch.equal(Fg, Fh)
    return h


@pytest.mark.parametrize("k", [0, 1, 2, 3, 4, 6])
@pytest.mark.parametrize("dims,stencil", [((9, 7, 5), 7), ((33, 3, 2), 7), ((32, 5, 3), 7), ((64, 4, 3), 7), ((8, 6, 5), 27), ((31, 1, 1), 7),
                                          ((1, 1, 1), 7)])
def test_grids(B, dims, stencil, k):
    rp, ci = grid_pattern(*dims, stencil)
    _same(B, dims[0] * dims[1] * dims[2], rp, ci, k)


@pytest.mark.parametrize("k", [0, 1, 2, 3])
@pytest.mark.parametrize("n,density,seed", [(32, 0.1, 1), (65, 0.05, 2), (300, 0.01, 3), (150, 0.08, 4)])
def test_nonsymmetric(B, n, density, seed, k):
    rp, ci = random_pattern(n, density=density, seed=seed)
    _same(B, n, rp, ci, k)


@pytest.mark.parametrize("width", [8, 9, 97, 385, 500])
def test_wide_rows(B, width):
    """Rows of `width` entries: both tables' limits, and past the large one (384 vertices)."""
    n = width + 5
    cols = [sorted(set(range(width)) | {i}) if i == width // 2 else sorted({i, width // 2}) for i in range(n)]
    rp = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int32)
    _same(B, n, rp, np.concatenate(cols).astype(np.int32), 1)


def test_row_capacity_limit(B):
    rp, ci = grid_pattern(7, 6, 5, 7)
    n, k = 210, 2
    widest = int(np.diff(B.bilu_symbolic(n, rp, ci, k).export()["row_ptr"]).max())
    _same(B, n, rp, ci, k, cap=widest)
    from paper_1703_01325_gb300 import _lib as L
    with pytest.raises(B.BiluError) as e:
        B.bilu_symbolic_gpu(n, rp, ci, k, row_capacity=widest - 1)
    assert e.value.status == L.BILU_ERR_OOM


@pytest.mark.parametrize("n,rp,ci", [
    (2, [0, 1, 2], [0, 0]),           # no diagonal
    (2, [0, 2, 3], [1, 0, 1]),        # unsorted
    (2, [0, 2, 3], [0, 0, 1]),        # twice
    (2, [0, 1, 2], [0, 2]),           # out of range
    (2, [0, 1, 2], [-1, 1]),
    (2, [1, 2, 3], [0, 1, 1]),        # row_ptr[0] != 0
    (3, [0, 2, 1, 3], [0, 1, 2]),     # descending row pointers
    (3, [0, 9, 2, 3], [0, 1, 2]),     # past the end
    (2, [0, 1, 1], [0]),              # an empty row
])
def test_malformed(B, n, rp, ci):
    from paper_1703_01325_gb300 import _lib as L
    with pytest.raises(B.BiluError) as e:
        B.bilu_symbolic_gpu(n, np.array(rp, np.int32), np.array(ci, np.int32), 1)
    assert e.value.status == L.BILU_ERR_PATTERN
