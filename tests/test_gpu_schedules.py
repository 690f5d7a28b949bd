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
