"""The factorization kernel where its batches end and its rows leave the staging
buffer, per block size: U rows of exactly a batch and one more (taken in slices),
rows on both sides of the buffer, the buffer left out (rows longer than it on
average, b >= 5).  FP64 against the oracle at the parity tests' tolerance, FP32 to
the bound of its sums."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1703_01325_gb300.reservoir import BlockSystem, random_block_values  # noqa: E402
from tests.gpu_util import TOL_FACTOR, OracleRun, device_system, rel_maxerr  # noqa: E402
from tests.oracle_helpers import diag_dominant_block_values  # noqa: E402

pytestmark = pytest.mark.gpu


def _blocks(widths, b, seed):
    """Full diagonal blocks of these widths, one row of each tied to the block before."""
    cols, at = [], 0
    for w in widths:
        cols += [set(range(at, at + w)) | ({at - 1} if at and i == at else set()) for i in range(at, at + w)]
        at += w
    cols = [sorted(c) for c in cols]
    rp = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int32)
    ci = np.concatenate(cols).astype(np.int32)
    rhs = random_block_values(at, b, seed=seed + 1)[:, :b].reshape(-1).copy()
    return BlockSystem(n=at, b=b, row_ptr=rp, col_idx=ci, vals=diag_dominant_block_values(at, b, rp, ci, seed), rhs=rhs)


@pytest.mark.parametrize("b,widths", [
    (1, (129, 3)), (1, (130, 7)), (1, (64, 65)), (2, (97, 2)), (2, (98, 40)),
    (3, (65, 5)), (3, (66, 64)), (3, (97,)), (3, (98, 9)), (4, (33, 34)), (4, (65, 66)),
    (5, (29, 30, 31)), (5, (32, 4)), (5, (43, 44)), (6, (29, 30)), (6, (33, 31)), (6, (43, 44, 2)),
    (7, (17, 18, 24)), (7, (25, 29, 30)), (7, (50, 3)), (8, (17, 18)), (8, (20, 21, 22)), (8, (24,)), (8, (25, 40)),
])
def test_batch_and_buffer_edges(libbilu, b, widths):
    _check(b, widths)


@pytest.mark.parametrize("rows", [17, 512, 1024])
@pytest.mark.parametrize("b", [1, 3, 5, 6, 7, 8])
def test_chunk_lengths(libbilu, b, rows):
    """The batch and the buffer shrink with the rows per chunk that shared memory also holds (1024: 8 KB)."""
    import paper_1703_01325_gb300.bilu as B
    old = B.bilu_get_factor_chunk()
    try:
        B.bilu_set_factor_chunk(rows)
        _check(b, (23, 22) * (30 if b < 5 else 24))
    finally:
        B.bilu_set_factor_chunk(old)


def _check(b, widths):
    import paper_1703_01325_gb300.bilu as B
    torch.cuda.set_device(0)
    S = _blocks(widths, b, seed=13 * b + sum(widths))
    o = OracleRun(S.n, b, S.row_ptr, S.col_idx, S.vals, 0)
    _, _, vals, _ = device_system(S, "cuda:0")
    P = B.bilu_symbolic(S.n, S.row_ptr, S.col_idx, 0).upload()
    F, info = B.bilu_factor(P, b, vals)
    F32, info32 = B.bilu_factor_f32(P, b, vals)
    assert info.status == 0 and info32.status == 0
    # FP32: each value is a sum of at most (width + 1) products of b terms, rounded at 2^-24
    tol32 = 8 * (max(widths) + 1) * b * 2.0 ** -24
    for tol, f in ((TOL_FACTOR, F), (tol32, F32.double())):
        for got, ref in zip((t.cpu().numpy() for t in B.factor_sections(P, b, f)), (o.L(), o.Dinv, o.U())):
            assert rel_maxerr(got, ref) <= tol
