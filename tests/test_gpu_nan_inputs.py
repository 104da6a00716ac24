"""Right-hand sides with NaN, infinities, signed zeros and the bit patterns the
kernels use as markers: every sweep schedule returns the same bits, and ends."""
import numpy as np
import pytest
import torch

import paper_0803_0048_gb300 as P
from paper_0803_0048_gb300 import _lib as L
from paper_0803_0048_gb300 import workloads as W

from gpu_helpers import assert_bits_equal, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


SCHEDS = [L.SCHED_FLAGS, L.SCHED_SINGLE_CTA, L.SCHED_CLUSTER, L.SCHED_WARP_CLUSTER,
          L.SCHED_WARP_CLUSTER_HELP]
PATTERNS = [0x7FF8000000000000, 0xFFF8000000000123, 0x7FF0000000000456, 0x7FF0DEADBEEFCAFE,
            0x7FF0000000000000, 0xFFF0000000000000, 0x8000000000000000]


@pytest.mark.parametrize("bits", PATTERNS, ids=[f"{b:016x}" for b in PATTERNS])
@pytest.mark.parametrize("diagonal", [False, True])
def test_schedules_agree(bits, diagonal):
    A = W.conv_diff(12, 2, (20.0, 20.0))
    if diagonal:
        i = np.arange(A.n)
        A = W.CSR(A.n, np.arange(A.n + 1, dtype=np.int64), i.astype(np.int32), 2.0 + 0.1 * i)
    rp, ci, av = to_dev(A)
    F = P.numeric(P.symbolic(rp, ci, 0), av)
    for row in (0, 40, A.n - 1):
        p = np.linspace(-1.0, 1.0, A.n)
        p.view(np.uint64)[row] = bits
        pd = torch.from_numpy(p).cuda()
        for transpose in (False, True):
            want = F.apply(pd, transpose=transpose, sched=L.SCHED_WARP_GRID)
            for s in SCHEDS:
                assert_bits_equal(F.apply(pd, transpose=transpose, sched=s), want,
                                  f"row {row} transpose {transpose} schedule {s}")
    assert F.status() == L.OK
