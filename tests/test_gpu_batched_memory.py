"""Memory of the batched solver's packed copies: bounded by an eighth of the free
memory, made only when a spinning schedule runs, and results that do not depend
on how many work slots have one."""
import numpy as np
import pytest
import torch

import paper_0803_0048_gb300 as P

from gpu_helpers import assert_bits_equal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def four_chains(n):
    """Rows i with the column i - 4 and its mirror: n / 4 levels of four rows,
    whose packed copy takes eight padded slots a row."""
    i = np.arange(n)
    ok = np.stack([i >= 4, np.ones(n, bool), i + 4 < n], 1)
    cols = np.stack([i - 4, i, i + 4], 1)
    rp = np.zeros(n + 1, np.int64)
    rp[1:] = np.cumsum(ok.sum(1))
    vals = np.tile([-1.0, 4.0, -1.0], (n, 1))
    return tuple(torch.from_numpy(a).cuda() for a in (rp, cols[ok].astype(np.int32), vals[ok]))


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def batch(n, count, schedule):
    rp, ci, v = four_chains(n)
    S = P.symbolic(rp, ci, 0)
    S.depth()
    x = torch.zeros(count, n, dtype=torch.float64, device="cuda")
    b = torch.rand(count, n, dtype=torch.float64, generator=torch.Generator().manual_seed(3)).cuda()
    items = [(S, v, b[t], x[t]) for t in range(count)]
    free = free_bytes()
    B = P.BatchSolve(items, restart=2, rtol=1e-8, maxit=2)
    made = free - free_bytes()
    if schedule is not None:
        B.set_schedule(*schedule)
    B.solve()
    return free, made, free - free_bytes(), x, B


def test_packed_copies_take_an_eighth_at_most():
    n, count = 100000, 608
    copy = 176 * 8 * n  # of one work slot: 85 GB in all
    buffers = (2 * n + 4 * (n + 1) + 4 * (3 * n)) * 8  # bases, vectors and F, generously
    free, made, after, *_ = batch(n, count, (256, 1))
    assert count * copy > free // 8 + count * buffers, "the case no longer exceeds the bound"
    assert made <= count * buffers
    assert after <= count * buffers + free // 8


def test_no_copies_for_the_level_barriers():
    n, count = 4000, 64
    _, _, after, x, B = batch(n, count, (256, 0))
    assert after < count * 176 * 8 * n // 2  # the copies would take 360 MB
    _, _, _, y, B2 = batch(n, count, (256, 1))
    assert_bits_equal(x, y, "barriers and spinning")
    assert [i.iters for i in B.results()] == [i.iters for i in B2.results()]
