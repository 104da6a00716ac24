"""Memory of the ring sweeps' plan: at most an eighth of what is free, else the
sweep runs as another kind, with the same bits."""
import numpy as np
import pytest
import torch

import paper_0803_0048_gb300 as P
from paper_0803_0048_gb300 import _lib as L

from gpu_helpers import assert_bits_equal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def chain(n):
    i = np.arange(n)
    cols = np.stack([i - 1, i, i + 1], 1)
    ok = (cols >= 0) & (cols < n)
    rp = np.zeros(n + 1, np.int64)
    rp[1:] = np.cumsum(ok.sum(1))
    vals = np.tile([-1.0, 3.0, -1.0], (n, 1))
    return tuple(torch.from_numpy(a).cuda() for a in (rp, cols[ok].astype(np.int32), vals[ok]))


def test_plan_takes_an_eighth_at_most():
    """800,000 levels of one row: 410 MB a direction, 3 GB free."""
    n = 800000
    rp, ci, v = chain(n)
    F = P.numeric(P.symbolic(rp, ci, 0), v)
    p = torch.rand(n, dtype=torch.float64, generator=torch.Generator().manual_seed(1)).cuda()
    want = F.apply(p, sched=L.SCHED_WARP_GRID)
    rest = torch.empty(free_bytes() - 3 * 10**9, dtype=torch.uint8, device="cuda")
    try:
        free = free_bytes()
        assert 16 * 32 * n > free // 8, "the case no longer exceeds the bound"
        for _ in range(2):
            assert_bits_equal(F.apply(p, sched=L.SCHED_SINGLE_CTA), want, "little memory")
        assert free - free_bytes() <= free // 8
    finally:
        del rest
        torch.cuda.empty_cache()
    F2 = P.numeric(P.symbolic(rp, ci, 0), v)
    assert_bits_equal(F2.apply(p, sched=L.SCHED_SINGLE_CTA), want, "with a plan")
