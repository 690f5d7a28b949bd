"""bilu_apply_info names the schedule and the warps an apply runs on: the general
solve schedule, or the second one that rows of one pass run on."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1703_01325_gb300.bilu as B  # noqa: E402
from paper_1703_01325_gb300.reservoir import grid_pattern, reservoir_system  # noqa: E402


def test_arguments_and_no_schedule(libbilu):
    P = B.bilu_symbolic(120, *grid_pattern(6, 5, 4, 7), 1)
    assert P.apply_info(3)["rows"] == 0 and P.apply_info(3, f32=True)["rows"] == 0
    for b in (0, 9):
        with pytest.raises(B.BiluError):
            P.apply_info(b)
    assert libbilu.bilu_apply_info(None, 3, 0, None, None) != 0
    assert libbilu.bilu_apply_info(P.handle, 3, 0, None, None) == 0


def test_warps_that_are_set_are_used(libbilu):
    """A 27-point ILU(2) row has up to 60 blocks a side: eight warps unless 4 is set."""
    rp, ci = grid_pattern(9, 8, 7, 27)
    P = B.bilu_symbolic(504, rp, ci, 2)
    try:
        B.bilu_set_trisolve_warps(0)
        assert [P.apply_info(b, f32=True)["warps"] for b in (1, 2, 3, 8)] == [4, 8, 8, 8]
        for w in (4, 8, 16):
            B.bilu_set_trisolve_warps(w)
            assert [P.apply_info(b)["warps"] for b in (1, 3, 8)] == [w] * 3
    finally:
        B.bilu_set_trisolve_warps(0)


@pytest.mark.gpu
@pytest.mark.parametrize("dims,b,k,f64,f32", [
    ((30, 30, 30), 3, 1, 60, 60),    # one pass: two lines
    ((30, 30, 30), 5, 0, 60, 60),
    ((30, 30, 30), 5, 1, 32, 32),    # two passes over four groups: the general schedule
    ((30, 30, 30), 3, 2, None, None),  # rows of more than eight blocks: no second schedule
    ((16, 30, 30), 3, 2, None, 32),  # wide rows of two passes, FP32: the two lines of the size rule
    ((16, 30, 30), 5, 2, None, None),  # three passes
    ((16, 30, 30), 8, 2, None, None),  # few rows per level
    ((70, 30, 10), 3, 1, 140, 32),   # lines above 64 rows: FP64 only
    ((70, 30, 10), 3, 0, 32, 32),    # and not for rows of four blocks and fewer
])
def test_which_schedule(libbilu, dims, b, k, f64, f32):
    """... and both schedules give the same bits."""
    torch.cuda.set_device(0)
    B.bilu_set_trisolve_warps(0)
    S = reservoir_system(*dims, b, sigma=1.0, accum=0.01, seed=2)
    vals, rhs = torch.from_numpy(S.vals.reshape(-1)).cuda(), torch.from_numpy(S.rhs).cuda()
    P = B.bilu_symbolic_gpu(S.n, S.row_ptr, S.col_idx, k).upload()
    general = P.schedule_info()["solve_rows"]
    assert general == B.bilu_auto_trisolve_chunk(P)
    assert [P.apply_info(b)["rows"], P.apply_info(b, f32=True)["rows"]] == [f64 or general, f32 or general]
    F, _ = B.bilu_factor(P, b, vals)
    F32 = B.bilu_convert_f32(F)
    x, x32 = B.bilu_apply(P, b, F, rhs), B.bilu_apply_f32(P, b, F32, rhs)
    old = B.bilu_get_trisolve_chunk()
    try:
        B.bilu_set_trisolve_chunk(general)
        P.reschedule()
    finally:
        B.bilu_set_trisolve_chunk(old)
    assert P.apply_info(b)["rows"] == P.apply_info(b, f32=True)["rows"] == general
    assert torch.equal(B.bilu_apply(P, b, F, rhs), x) and torch.equal(B.bilu_apply_f32(P, b, F32, rhs), x32)


@pytest.mark.gpu
def test_large_blocks_with_many_rows_per_level(libbilu):
    """120x80x35 ILU(2): 565 rows per level, more than the 456 lines that three CTAs on each of 152 SMs hold, where
    the size rule cuts two lines: FP64 rows of b >= 7 and FP32 rows of two passes run on two lines."""
    torch.cuda.set_device(0)
    B.bilu_set_trisolve_warps(0)
    P = B.bilu_symbolic_gpu(336000, *grid_pattern(120, 80, 35, 7), 2).upload()
    assert P.schedule_info()["solve_rows"] == 120
    assert [P.apply_info(b)["rows"] for b in (1, 3, 6, 7, 8)] == [120, 120, 120, 240, 240]
    assert [P.apply_info(b, f32=True)["rows"] for b in (1, 4, 5, 8)] == [240, 240, 120, 120]


@pytest.mark.gpu
@pytest.mark.parametrize("dims,wide,narrow", [((60, 50, 40), (2, 3, 4, 5, 6), (8,)), ((40, 40, 20), (2, 3, 4, 5, 6, 7, 8), ())])
def test_eight_warps_while_enough_lines_are_resident(libbilu, dims, wide, narrow):
    """27-point ILU(2) rows: 136 and 64 rows per level, on 152 SMs with three, two (b >= 4) or one (b >= 7)
    eight-warp CTA each."""
    torch.cuda.set_device(0)
    B.bilu_set_trisolve_warps(0)
    n = dims[0] * dims[1] * dims[2]
    P = B.bilu_symbolic_gpu(n, *grid_pattern(*dims, 27), 2).upload()
    assert all(P.apply_info(b)["warps"] == 8 for b in wide) and all(P.apply_info(b)["warps"] == 4 for b in narrow)
    assert all(P.apply_info(b, f32=True)["warps"] == 8 for b in wide + narrow)


@pytest.mark.gpu
@pytest.mark.parametrize("host", [True, False])
def test_lines_of_all_lengths_take_the_general_schedule(libbilu, host):
    """A grid whose lines lost cells at their ends has lines of 20 to 30 rows, most of them of 30."""
    torch.cuda.set_device(0)
    B.bilu_set_trisolve_warps(0)
    rp, ci = grid_pattern(30, 30, 30, 7)
    rng = np.random.default_rng(4)
    lost = np.where(rng.random(900) < 0.4, rng.integers(1, 11, 900), 0)
    keep = np.arange(27000) % 30 < 30 - np.repeat(lost, 30)
    new, rows = np.cumsum(keep) - 1, np.repeat(np.arange(27000), np.diff(rp))
    ok = keep[rows] & keep[ci]
    n = int(keep.sum())
    rp = np.concatenate([[0], np.cumsum(np.bincount(new[rows[ok]], minlength=n))]).astype(np.int32)
    ci = new[ci[ok]].astype(np.int32)
    P = (B.bilu_symbolic(n, rp, ci, 1) if host else B.bilu_symbolic_gpu(n, rp, ci, 1)).upload()
    assert P.apply_info(3)["rows"] == P.apply_info(3, f32=True)["rows"] == P.schedule_info()["solve_rows"]
