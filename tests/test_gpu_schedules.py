"""Building schedules with little device memory, and for patterns whose chunks
have many predecessors: what is not needed is not asked for, and what cannot be
had is done without where there is another way."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1703_01325_gb300.bilu as B  # noqa: E402
from paper_1703_01325_gb300.reservoir import grid_pattern, random_pattern  # noqa: E402

pytestmark = pytest.mark.gpu

KEYS = ("bounds", "ord_lower", "ord_upper", "tick_lower", "tick_upper")


@pytest.fixture(autouse=True)
def _device(libbilu):
    torch.cuda.set_device(0)
    yield
    B.bilu_test_fail_alloc(0)


def _same_schedule(g, h, rows):
    a, b = g.schedule(rows), h.schedule(rows)
    for key in KEYS:
        assert np.array_equal(a[key], b[key]), key


@pytest.mark.parametrize("rows,limit", [
    (1, 3 << 20),      # 24000 chunks: 64 words each would be 6 MB
    (8, 700 << 10),    # 3000 chunks: 0.8 MB that cannot be had; the rest needs at most 0.4 MB at once
])
def test_lists_of_any_length_instead(rows, limit):
    rp, ci = grid_pattern(40, 30, 20, 7)
    g, h = B.bilu_symbolic_gpu(24000, rp, ci, 0), B.bilu_symbolic(24000, rp, ci, 0)
    B.bilu_test_fail_alloc(limit)
    _same_schedule(g, h, rows)


@pytest.mark.parametrize("n,density,rows", [(4000, 0.01, 16), (4000, 0.01, 32), (900, 0.08, 8)])
def test_many_predecessors(n, density, rows):
    """Every chunk depends on more chunks than the gathered lists hold (64); some before 65 rows of work."""
    rp, ci = random_pattern(n, density=density, seed=n + rows)
    _same_schedule(B.bilu_symbolic_gpu(n, rp, ci, 0, row_capacity=1024), B.bilu_symbolic(n, rp, ci, 0), rows)


def _apply_of(P):
    """Status and result of an apply (b = 3) with fixed factors and right-hand side."""
    g = torch.Generator().manual_seed(1)
    F = (torch.rand(P.factor_bytes(3) // 8, generator=g, dtype=torch.float64) * 0.01).cuda()
    return B.bilu_apply(P, 3, F, torch.rand(27000 * 3, generator=g, dtype=torch.float64).cuda()).clone()


def test_second_schedule_is_left_out_without_memory(libbilu):
    """A 30^3 ILU(1) grid: 226 KB the general schedule, 223 KB each of its two gathered lists, 221 KB the second
    schedule (which fails), 112 KB the factorization's."""
    P = B.bilu_symbolic_gpu(27000, *grid_pattern(30, 30, 30, 7), 1)
    B.bilu_test_fail_alloc(215 << 10, 3)
    P.upload()
    assert P.schedule_info() == {"solve_rows": 32, "factor_rows": 60} and P.apply_info(3)["rows"] == 32
    x = _apply_of(P)
    B.bilu_test_fail_alloc(0)
    P.reschedule()
    assert P.apply_info(3)["rows"] == 60
    assert torch.equal(_apply_of(P), x)


def test_failed_reschedule_leaves_all_old_schedules(libbilu):
    """The factorization's schedule fails (the sixth allocation of 100 KB and more: two of row gaps, the general
    schedule, its two gathered lists, this): no schedule of the new setting is in place."""
    from paper_1703_01325_gb300 import _lib as L
    P = B.bilu_symbolic_gpu(27000, *grid_pattern(30, 30, 30, 7), 1).upload()
    before = (P.schedule_info(), P.apply_info(3), P.apply_info(6))
    x = _apply_of(P)
    try:
        B.bilu_set_trisolve_chunk(40)
        B.bilu_test_fail_alloc(100 << 10, 5)
        with pytest.raises(B.BiluError) as e:
            P.reschedule()
        assert e.value.status == L.BILU_ERR_OOM
        assert (P.schedule_info(), P.apply_info(3), P.apply_info(6)) == before
        assert torch.equal(_apply_of(P), x)
        B.bilu_test_fail_alloc(0)
        P.reschedule()
        assert P.schedule_info()["solve_rows"] == P.apply_info(3)["rows"] == 40
        assert torch.equal(_apply_of(P), x)
    finally:
        B.bilu_set_trisolve_chunk(0)


@pytest.mark.parametrize("dims,k,allocs", [((16, 16, 8), 1, 3), ((8, 6, 5), 0, 2), ((8, 8, 6), 2, 2)])
def test_small_host_patterns_take_the_host_builder(libbilu, dims, k, allocs):
    """Small patterns completed on the host need one allocation per schedule (general, factorization and, for lines
    of 16 rows and more, the second one), and run as the same pattern completed on the device."""
    rp, ci = grid_pattern(*dims, 7)
    n = int(np.prod(dims))
    h, g = B.bilu_symbolic(n, rp, ci, k), B.bilu_symbolic_gpu(n, rp, ci, k).upload()
    B.bilu_test_fail_alloc(1, allocs)
    h.upload()
    B.bilu_test_fail_alloc(0)
    assert (h.schedule_info(), h.apply_info(3)) == (g.schedule_info(), g.apply_info(3))
    gen = torch.Generator().manual_seed(1)
    F = (torch.rand(h.factor_bytes(3) // 8, generator=gen, dtype=torch.float64) * 0.01).cuda()
    r = torch.rand(3 * n, generator=gen, dtype=torch.float64).cuda()
    assert torch.equal(B.bilu_apply(h, 3, F, r), B.bilu_apply(g, 3, F, r))
