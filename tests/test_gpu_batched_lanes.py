"""The batched numeric phase with a row per lane (wide levels of short rows)
against the oracle, bit for bit, where it can go wrong: the longest rows a lane
takes and one more, levels that end inside a warp, exactly as wide as the rule's
line and one row narrower, and several passes of the warps over a level; and
failures reported for their item with the smallest row."""
import numpy as np
import pytest
import torch

import oracle
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


def blocks(count, size):
    """`count` independent dense blocks: `size` levels of `count` rows."""
    rng = np.random.default_rng(100 * count + size)
    rp, ci, va = [0], [], []
    for b in range(count):
        for i in range(size):
            ci += list(range(b * size, (b + 1) * size))
            row = rng.uniform(-1, 1, size)
            row[i] = size + 1.0
            va += list(row)
            rp.append(len(ci))
    return W.CSR(count * size, np.array(rp, np.int64), np.array(ci, np.int32), np.array(va))


def systems():
    out = [(blocks(c, s), 0) for c, s in ((100, 1), (47, 2), (48, 2), (65, 7), (300, 15),
                                          (300, 16), (300, 17))]
    return out + [(W.conv_diff(20, 3, (50.0, 50.0, 50.0)), 1),
                  (W.conv_diff(24, 3, (50.0, 50.0, 50.0)), 0)]


def items_of(mats):
    items = []
    for A, k in mats:
        rp, ci, av = to_dev(A)
        b = torch.linspace(-1.0, 1.0, A.n, dtype=torch.float64, device="cuda")
        items.append((P.symbolic(rp, ci, k), av, b, torch.zeros_like(b)))
    return items


@pytest.mark.parametrize("width", [256, 512, 1024])
def test_lane_rows_bit_exact(width):
    mats = systems()
    items = items_of(mats)
    B = P.BatchSolve(items, restart=30, rtol=1e-8)
    B.set_schedule(width, True)
    B.solve()
    for (A, k), (_, _, b, x), r in zip(mats, items, B.results()):
        F = oracle.factor(A, k)
        st, xo, it, rel, cyc = oracle.gmres(A.n, A.rowptr, A.colind, A.val, b.cpu().numpy(),
                                            oracle.PREC_ILU, (F["rowptr"], F["colind"], F["val"]),
                                            30, 1e-8, dotmode=oracle.DOT_TREE)
        assert st == 0 and (r.iters, r.cycles) == (it, cyc)
        assert r.status == 0
        assert_bits_equal(x, xo, f"n = {A.n}")


@pytest.mark.parametrize("width", [256, 512, 1024])
def test_lane_rows_report_failures(width):
    mats = systems()
    items = items_of(mats)
    A = mats[5][0]
    items[5][1][int(A.rowptr[777])] = float("nan")
    items[3][1].zero_()
    B = P.BatchSolve(items, restart=30, rtol=1e-8)
    B.set_schedule(width, True)
    B.solve()
    res = B.results()
    assert res[5].status == L.ENONFINITE and res[5].row == 777
    assert res[3].status == L.EZEROPIVOT and res[3].row == 0
    assert all(r.status == 0 for i, r in enumerate(res) if i not in (3, 5))
