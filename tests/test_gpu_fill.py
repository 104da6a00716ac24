"""The symbolic phase level by level (no waits between rows) against the oracle:
patterns whose window it does not take (these keep the walk with waits), and
patterns whose stored diagonals are incomplete."""
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


def _wide_window(n=66000):
    """A tridiagonal matrix whose first row also reaches the last column: the
    rows' window is wider than the passes over fill levels take, so k >= 2 runs
    both phases in one launch (the walk with waits)."""
    rp, ci, va = [0], [], []
    for i in range(n):
        cols = [c for c in (i - 1, i, i + 1) if 0 <= c < n]
        if i == 0:
            cols.append(n - 1)
        ci += cols
        va += [4.0 if c == i else -1.0 for c in cols]
        rp.append(len(ci))
    return W.CSR(n, np.array(rp, np.int64), np.array(ci, np.int32), np.array(va))


@pytest.mark.parametrize("k", [1, 2, 3])
def test_symbolic_wide_window(k):
    A = _wide_window()
    rp, ci, av = to_dev(A)
    ref = oracle.factor(A, k)
    for S, F in (P.factor(rp, ci, av, k), (lambda S: (S, P.numeric(S, av)))(P.symbolic(rp, ci, k))):
        grp, gci, glev, gdg = [t.cpu().numpy() for t in S.pattern()]
        assert np.array_equal(grp, ref["rowptr"]) and np.array_equal(gci, ref["colind"])
        assert np.array_equal(glev, ref["level"])
        assert_bits_equal(F.values(), ref["val"], "factor values")


@pytest.mark.parametrize("k", [2, 3, 5])
@pytest.mark.parametrize("n,dens,seed", [(33, 0.2, 31), (400, 0.02, 32), (1500, 0.003, 33)])
def test_symbolic_passes_without_stored_diagonals(n, dens, seed, k):
    """Fill level by level on patterns with diagonals missing from A (some
    enter as fill): pattern, levels and the first row still without one as
    the oracle's."""
    A = W.random_sparse(n, dens, seed)
    keep = np.ones(A.nnz, dtype=bool)
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    keep[(A.colind == rows) & (rows % 7 == 3)] = False
    rp = np.zeros(A.n + 1, dtype=np.int64)
    rp[1:] = np.cumsum(np.bincount(rows[keep], minlength=A.n))
    B = W.CSR(A.n, rp, A.colind[keep].copy(), A.val[keep].copy())
    drp, dci, _ = to_dev(B)
    st, bad, *rest = oracle.symbolic(B.n, B.rowptr, B.colind, k)
    if st == oracle.OK:
        got = [t.cpu().numpy() for t in P.symbolic(drp, dci, k).pattern()]
        for g, want in zip(got, rest[:3]):
            assert np.array_equal(g, want)
    else:
        with pytest.raises(P.IlukError) as e:
            P.symbolic(drp, dci, k)
        assert e.value.status == L.ENODIAG and e.value.row == bad
