"""The update plan at its limits, with the path that ran told by the launches the
plan's making takes: the longest dense row it takes and one more entry, more than
32 (64, 96) pivots a row, rows of 128 and 129 entries, rows of 2,048 and 2,049
updates.  Bit for bit against the oracle, first factorization and kept plan."""
import numpy as np
import pytest
import torch

import oracle
import paper_0803_0048_gb300 as P
from paper_0803_0048_gb300 import workloads as W

from gpu_helpers import assert_bits_equal, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def groups(count, extra, dense):
    """`count` independent groups: `extra` rows of a diagonal and an entry in
    the group's last column, then a dense block of `dense` rows whose last
    row also has the extra columns.  That row: extra + dense entries, extra +
    dense (dense - 1) / 2 updates."""
    rng = np.random.default_rng(extra * 1000 + dense)
    size = extra + dense
    rp, ci, va = [0], [], []
    for g in range(count):
        base = g * size
        last = base + size - 1
        for i in range(size):
            if i < extra:
                cols = [base + i] + ([last] if base + i != last else [])
            else:
                cols = list(range(base + extra, base + size))
                if i == size - 1:
                    cols = list(range(base, base + extra)) + cols
            row = rng.uniform(-1, 1, len(cols))
            row[cols.index(base + i)] = len(cols) + 1.0
            ci += cols
            va += list(row)
            rp.append(len(ci))
    return W.CSR(count * size, np.array(rp, np.int64), np.array(ci, np.int32), np.array(va))


# launches of the plan's making: its count pass, a scan (three), its write pass
NONE, COUNTED, PLANNED = 0, 4, 5


@pytest.mark.parametrize("extra,dense,made", [
    (0, 2, PLANNED), (0, 33, PLANNED), (0, 34, PLANNED), (0, 64, PLANNED), (0, 65, COUNTED),
    (31, 2, PLANNED), (32, 1, PLANNED), (64, 34, PLANNED), (127, 1, PLANNED), (128, 1, NONE),
    (94, 34, PLANNED), (95, 34, NONE), (32, 64, PLANNED), (33, 64, COUNTED)])
def test_plan_limits(extra, dense, made):
    A = groups(60, extra, dense)
    rp, ci, av = to_dev(A)
    S = P.symbolic(rp, ci, 0)
    assert S.max_row == extra + dense
    S.depth()  # the level orders, so that the calls below differ by the plan alone
    counts = [P.launch_count()]
    F = P.numeric(S, av)
    counts.append(P.launch_count())
    F2 = P.numeric(S, av)
    counts.append(P.launch_count())
    assert (counts[1] - counts[0]) - (counts[2] - counts[1]) == made
    ref = oracle.factor(A, 0)
    assert_bits_equal(F.values(), ref["val"], "first")
    assert_bits_equal(F2.values(), ref["val"], "second")
    F.refactor(av * -0.75)
    r = oracle.factor(W.CSR(A.n, A.rowptr, A.colind, A.val * -0.75), 0)
    assert_bits_equal(F.values(), r["val"], "refactored")
