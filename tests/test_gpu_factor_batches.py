"""The factorization kernel at the edges of its batches: pivots whose U rows
are longer than a batch holds (taken in slices), more than 32 pivots per row,
rows wider than the staging buffer (worked on in place), rows without pivots.
Dense trailing blocks give the widest rows; FP64 against the oracle at the
parity tests' tolerance, FP32 against the same to the FP32 bound of the sums."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1703_01325_gb300.reservoir import BlockSystem, random_block_values  # noqa: E402
from tests.gpu_util import TOL_FACTOR, OracleRun, device_system, rel_maxerr  # noqa: E402
from tests.oracle_helpers import diag_dominant_block_values  # noqa: E402

pytestmark = pytest.mark.gpu


def _block_dense(n, width, b, seed):
    """Rows of a diagonal block of `width` rows are full; a chain links the blocks."""
    cols = [sorted({j for j in range(i - i % width, min(n, i - i % width + width))} | ({i - 1} if i else set()))
            for i in range(n)]
    rp = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int32)
    ci = np.concatenate(cols).astype(np.int32)
    vals = diag_dominant_block_values(n, b, rp, ci, seed)
    rhs = random_block_values(n, b, seed=seed + 1)[:, :b].reshape(-1).copy()
    return BlockSystem(n=n, b=b, row_ptr=rp, col_idx=ci, vals=vals, rhs=rhs)


@pytest.mark.parametrize("width", [1, 12, 13, 25, 34, 49, 66, 100])
@pytest.mark.parametrize("b", [1, 3, 4, 6, 8])
def test_factor_row_widths(libbilu, b, width):
    import paper_1703_01325_gb300.bilu as B
    torch.cuda.set_device(0)
    S = _block_dense(2 * width + 3, width, b, seed=7 * b + width)
    o = OracleRun(S.n, b, S.row_ptr, S.col_idx, S.vals, 0)
    _, _, vals, _ = device_system(S, "cuda:0")
    P = B.bilu_symbolic(S.n, S.row_ptr, S.col_idx, 0).upload()
    F, info = B.bilu_factor(P, b, vals)
    F32, info32 = B.bilu_factor_f32(P, b, vals)
    assert info.status == 0 and info32.status == 0
    # FP32: each value is a sum of at most (width + 1) products of b terms, rounded at 2^-24
    tol32 = 8 * (width + 1) * b * 2.0 ** -24
    for tol, f in ((TOL_FACTOR, F), (tol32, F32.double())):
        for got, ref in zip((t.cpu().numpy() for t in B.factor_sections(P, b, f)), (o.L(), o.Dinv, o.U())):
            assert rel_maxerr(got, ref) <= tol
