"""The variants of the sweeps' row kernel and the schedules they run on, at the
row widths where the dispatch changes: one to five passes over the groups (the
waits joined or not), 40 blocks and more in four passes (eight warps per CTA),
grids of whole lines on one, two or three lines per chunk.  FP64 against the
oracle; FP32 against the oracle on the rounded factors, to the bound of its sums."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1703_01325_gb300.reservoir import BlockSystem, random_block_values, reservoir_system  # noqa: E402
from tests.gpu_util import TOL_APPLY, OracleRun, device_system, rel_maxerr  # noqa: E402
from tests.oracle_helpers import diag_dominant_block_values  # noqa: E402

pytestmark = pytest.mark.gpu


def _check(S, k):
    import paper_1703_01325_gb300.bilu as B
    torch.cuda.set_device(0)
    b = S.b
    o = OracleRun(S.n, b, S.row_ptr, S.col_idx, S.vals, k)
    _, _, vals, rhs = device_system(S, "cuda:0")
    P = B.bilu_symbolic(S.n, S.row_ptr, S.col_idx, k).upload()
    F, info = B.bilu_factor(P, b, vals)
    assert info.status == 0
    for r in (rhs, rhs * 0.5):
        work = B.workspace(P.apply_workspace_bytes(b))
        x = B.bilu_apply(P, b, F, r, work=work)
        assert B.bilu_workspace_status(work) == 0
        assert rel_maxerr(x.cpu().numpy(), o.apply(r.cpu().numpy())) <= TOL_APPLY
    x32 = B.bilu_apply_f32(P, b, B.bilu_convert_f32(F), rhs).cpu().numpy()
    # each row sums at most (width + 1) products of b terms, rounded at 2^-24
    width = int(np.diff(o.prp).max())
    assert rel_maxerr(x32, o.apply(S.rhs)) <= 16 * (width + 1) * b * 2.0 ** -24


@pytest.mark.parametrize("blocks", [1, 4, 8, 9, 16, 17, 33, 39, 40, 41, 64, 70])
@pytest.mark.parametrize("b", [1, 2, 3, 4, 5, 8])
def test_row_widths(libbilu, b, blocks):
    """Full rows of up to `blocks` blocks beside the diagonal, in a dense band."""
    n = 2 * blocks + 7
    cols = [list(range(max(0, i - blocks), min(n, i + blocks + 1))) for i in range(n)]
    rp = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int32)
    ci = np.concatenate(cols).astype(np.int32)
    vals = diag_dominant_block_values(n, b, rp, ci, 11 * b + blocks)
    rhs = random_block_values(n, b, seed=blocks)[:, :b].reshape(-1).copy()
    _check(BlockSystem(n=n, b=b, row_ptr=rp, col_idx=ci, vals=vals, rhs=rhs), 0)


@pytest.mark.parametrize("dims", [(16, 9, 6), (17, 12, 5), (40, 7, 5), (19, 3, 20)])
@pytest.mark.parametrize("b,k,stencil", [(2, 0, 7), (3, 1, 7), (5, 0, 7), (6, 1, 7), (3, 1, 27), (2, 2, 27)])
def test_grid_lines(libbilu, dims, b, k, stencil):
    _check(reservoir_system(*dims, b, stencil=stencil, sigma=1.0, accum=0.01, seed=5), k)
