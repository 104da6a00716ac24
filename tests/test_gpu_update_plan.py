"""The numeric phase on an update plan (wide DAGs of short rows) against the
oracle, bit for bit, where it can go wrong: rows of exactly the longest length
it takes and one more, more than 32 pivots a row, rows without pivots, pivots
without updates, refactorization with new values on the kept plan, a zero pivot
and a non-finite value on it, and a withheld row running out its wait."""
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
    """`count` independent dense blocks: rows of `size` entries, levels `count`
    rows wide, size - 1 pivots in a block's last row."""
    rng = np.random.default_rng(size)
    rp, ci, va = [0], [], []
    for b in range(count):
        for i in range(size):
            ci += list(range(b * size, (b + 1) * size))
            row = rng.uniform(-1, 1, size)
            row[i] = size + 1.0
            va += list(row)
            rp.append(len(ci))
    return W.CSR(count * size, np.array(rp, np.int64), np.array(ci, np.int32), np.array(va))


CASES = [("diagonal", blocks(300, 1), 0), ("pairs", blocks(64, 2), 0), ("dense33", blocks(64, 33), 0),
         ("dense65", blocks(50, 65), 0), ("dense66", blocks(50, 66), 0),
         ("poisson27_24_k1", W.poisson27(24), 1),
         ("convdiff3d_24_k2", W.conv_diff(24, 3, (50.0, 50.0, 50.0)), 2),
         ("convdiff3d_24_k0", W.conv_diff(24, 3, (50.0, 50.0, 50.0)), 0),
         ("convdiff2d_200_k2", W.conv_diff(200, 2, (20.0, 20.0)), 2)]


@pytest.mark.parametrize("name,A,k", CASES, ids=[c[0] for c in CASES])
def test_refactor_bit_exact(name, A, k):
    rp, ci, av = to_dev(A)
    S = P.symbolic(rp, ci, k)
    F = P.numeric(S, av)
    ref = oracle.factor(A, k)
    assert_bits_equal(F.values(), ref["val"], name)
    for scale in (1.5, -0.75):
        F.refactor(av * scale)
        r = oracle.factor(W.CSR(A.n, A.rowptr, A.colind, A.val * scale), k)
        assert_bits_equal(F.values(), r["val"], f"{name} scale {scale}")


def test_failures_on_a_plan():
    A = W.poisson27(14)
    rp, ci, av = to_dev(A)
    S = P.symbolic(rp, ci, 0)
    F = P.numeric(S, av)
    row = 1500
    bad = av.clone()
    bad[int(A.rowptr[row])] = float("nan")
    with pytest.raises(P.IlukError) as e:
        F.refactor(bad)
    assert e.value.status == L.ENONFINITE and e.value.row == row
    zero = torch.zeros_like(av)
    with pytest.raises(P.IlukError) as e:
        F.refactor(zero)
    assert e.value.status == L.EZEROPIVOT and e.value.row == 0
    old = P.set_wait_limit(20_000_000)
    P.debug_hold_row(100)
    try:
        with pytest.raises(P.IlukError) as e:
            F.refactor(av)
        assert e.value.status == L.ETIMEOUT
    finally:
        P.debug_hold_row(-1)
        P.set_wait_limit(old)
    F.refactor(av)  # the context is still healthy
    assert_bits_equal(F.values(), oracle.factor(A, 0)["val"], "after the failures")
