"""Ring sweeps (SINGLE_CTA and CLUSTER) in which rows read row 0, and its
neighbours, from beyond the ring while the ring's last entry is still empty:
cyclic bands, periodic grids, a filled first column, a few late rows over many
independent ones.  Bit for bit against the oracle, both directions, plain and
transposed, and through the one-call solve, which picks these sweeps by itself."""
import numpy as np
import pytest
import torch

import oracle
import paper_0803_0048_gb300 as P
from paper_0803_0048_gb300 import _lib as L
from paper_0803_0048_gb300 import workloads as W

from gpu_helpers import assert_bits_equal, to_dev, vec

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def from_rows(rows, seed):
    """Off-diagonal columns per row, random values, a dominant diagonal."""
    rng = np.random.default_rng(seed)
    rp, ci, va = [0], [], []
    for i, r in enumerate(rows):
        cols = sorted(set(r) | {i})
        ci += cols
        va += [float(len(cols)) + 1.0 if c == i else rng.uniform(-1, 1) for c in cols]
        rp.append(len(ci))
    return W.CSR(len(rows), np.array(rp, np.int64), np.array(ci, np.int32), np.array(va))


def cyclic(n):
    return [[(i - 1) % n, (i + 1) % n] for i in range(n)]


def periodic(N):
    return [[y * N + (x - 1) % N, y * N + (x + 1) % N, (y - 1) % N * N + x, (y + 1) % N * N + x]
            for y in range(N) for x in range(N)]


def first_column(n, cols=(0,)):
    """Tridiagonal with filled first columns."""
    return [[j for j in (i - 1, i + 1) if 0 <= j < n] + [c for c in cols if c < i]
            for i in range(n)]


def late_rows(n, late, transposed):
    """n - late rows of a diagonal only, then `late` rows that read column 0."""
    rows = [[] for _ in range(n)]
    for i in range(n - late, n):
        if transposed:
            rows[0].append(i)  # column 0 of the transpose
        else:
            rows[i].append(0)
    return rows


CASES = [(f"cyclic{n}", cyclic(n), 0) for n in (192, 193, 200, 256, 257)]
CASES += [("cyclic200_k2", cyclic(200), 2),
          ("periodic100", periodic(100), 0),
          ("periodic100_k1", periodic(100), 1),
          ("first_column400", first_column(400), 0),
          ("first_columns400", first_column(400, (0, 1, 2, 31)), 0),
          ("late_rows8000", late_rows(8000, 1000, False), 0),
          ("late_rows6160", late_rows(6160, 16, False), 0)]


@pytest.mark.parametrize("name,rows,k", CASES, ids=[c[0] for c in CASES])
@pytest.mark.parametrize("sched", [L.SCHED_SINGLE_CTA, L.SCHED_CLUSTER])
def test_far_first_rows_bit_exact(name, rows, k, sched):
    A = from_rows(rows, 3)
    rp, ci, av = to_dev(A)
    F = P.numeric(P.symbolic(rp, ci, k), av)
    ref = oracle.factor(A, k)
    trp, tci, tv = oracle.transpose(A.n, ref["rowptr"], ref["colind"], ref["val"])
    for rep in range(2):
        p, pd = vec(50 + rep, A.n)
        assert_bits_equal(F.apply(pd, sched=sched),
                          oracle.apply(A.n, ref["rowptr"], ref["colind"], ref["val"], p), name)
        assert_bits_equal(F.apply(pd, transpose=True, sched=sched),
                          oracle.apply_t(A.n, trp, tci, tv, p), name + " transposed")
    assert F.status() == L.OK


def test_far_first_row_of_the_transpose():
    """Rows that read far ahead in F, and far back in its transpose; row 0 of F
    is too long for a lane, so only the transposed forward sweep is a ring sweep."""
    n = 8000
    A = from_rows(late_rows(n, 1000, True), 4)
    rp, ci, av = to_dev(A)
    F = P.numeric(P.symbolic(rp, ci, 0), av)
    ref = oracle.factor(A, 0)
    trp, tci, tv = oracle.transpose(A.n, ref["rowptr"], ref["colind"], ref["val"])
    p, pd = vec(60, n)
    for sched in (L.SCHED_SINGLE_CTA, L.SCHED_CLUSTER):
        assert_bits_equal(F.apply(pd, sched=sched),
                          oracle.apply(n, ref["rowptr"], ref["colind"], ref["val"], p), "plain")
        assert_bits_equal(F.apply(pd, transpose=True, sched=sched),
                          oracle.apply_t(n, trp, tci, tv, p), "transposed")


@pytest.mark.parametrize("name", ["cyclic200", "periodic100", "late_rows8000"])
def test_one_call_solve_on_far_first_rows(name):
    """The schedule the one-call solve picks gives the oracle's iterations and x."""
    rows = dict((c[0], c[1]) for c in CASES)[name]
    A = from_rows(rows, 5)
    rp, ci, av = to_dev(A)
    b, bd = vec(70, A.n)
    ref = oracle.factor(A, 0)
    st, xo, it, rel, cyc = oracle.gmres(A.n, A.rowptr, A.colind, A.val, b, oracle.PREC_ILU,
                                        (ref["rowptr"], ref["colind"], ref["val"]), 20, 1e-10,
                                        dotmode=oracle.DOT_TREE)
    x, info = P.solve(rp, ci, av, bd, 0, restart=20, rtol=1e-10)
    assert st == oracle.OK and (info.iters, info.cycles) == (it, cyc)
    assert_bits_equal(x, xo, name)
