"""Patterns whose forward and backward sweeps have different DAGs (one-sided
upwind and bidiagonal matrices): each direction's schedule follows from its own
DAG, in the one-call solve and in the autotuner, plain and transposed, and the
results are the oracle's bit for bit."""
import numpy as np
import pytest
import torch

import oracle
import paper_0803_0048_gb300 as P
from paper_0803_0048_gb300 import _lib as L
from paper_0803_0048_gb300 import workloads as W

from gpu_helpers import assert_bits_equal, to_dev, vec

pytestmark = pytest.mark.gpu

FEW_SMS = (L.SCHED_SINGLE_CTA, L.SCHED_CLUSTER, L.SCHED_WARP_CLUSTER, L.SCHED_WARP_CLUSTER_HELP)
ALL_SMS = (L.SCHED_FLAGS, L.SCHED_WARP_GRID)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def from_rows(n, rows, seed):
    rng = np.random.default_rng(seed)
    rp, ci, va = [0], [], []
    for i in range(n):
        cols = sorted({j for j in rows(i) if 0 <= j < n} | {i})
        ci += cols
        va += [float(len(cols)) + 1.0 if c == i else rng.uniform(-1, 1) for c in cols]
        rp.append(len(ci))
    return W.CSR(n, np.array(rp, np.int64), np.array(ci, np.int32), np.array(va))


def upwind(N, sign):
    """A 2D grid whose rows read their two neighbours on one side only."""
    def rows(i):
        x = i % N + sign
        return ([i + sign] if 0 <= x < N else []) + [i + sign * N]
    return from_rows(N * N, rows, 1)


def kinds(sched):
    """(forward, backward) kinds of a packed pair."""
    f, b = sched & 0xFF, (sched >> 8) & 0xFF
    return f & 0xF, (b or f) & 0xF


@pytest.mark.parametrize("sign", [-1, 1])
def test_one_call_pick_per_direction(sign):
    A = upwind(256, sign)
    rp, ci, av = to_dev(A)
    b, bd = vec(80, A.n)
    x, info, (S, F) = P.solve(rp, ci, av, bd, 0, return_factors=True)
    deep, flat = kinds(F.schedule())[::-sign]
    assert S.depth()[::-sign] == (511, 1)
    assert deep in (L.SCHED_SINGLE_CTA, L.SCHED_CLUSTER) and flat in ALL_SMS
    ref = oracle.factor(A, 0)
    st, xo, it, *_ = oracle.gmres(A.n, A.rowptr, A.colind, A.val, b, oracle.PREC_ILU,
                                  (ref["rowptr"], ref["colind"], ref["val"]), 30, 1e-8,
                                  dotmode=oracle.DOT_TREE)
    assert st == oracle.OK and info.iters == it
    assert_bits_equal(x, xo, f"upwind {sign}")


@pytest.mark.parametrize("sign", [-1, 1])
def test_autotuner_per_direction(sign):
    """A bidiagonal matrix: one sweep is a chain of 6,000 rows (a few SMs take
    it in about half the time that all SMs need), the other has one level."""
    A = from_rows(6000, lambda i: [i + sign], 2)
    rp, ci, av = to_dev(A)
    F = P.numeric(P.symbolic(rp, ci, 0), av)
    p, pd = vec(81, A.n)
    ref = oracle.factor(A, 0)
    trp, tci, tv = oracle.transpose(A.n, ref["rowptr"], ref["colind"], ref["val"])
    assert_bits_equal(F.apply(pd),
                      oracle.apply(A.n, ref["rowptr"], ref["colind"], ref["val"], p), "plain")
    deep, flat = kinds(F.schedule())[::-sign]
    assert deep in FEW_SMS and flat in ALL_SMS
    assert_bits_equal(F.apply(pd, transpose=True), oracle.apply_t(A.n, trp, tci, tv, p),
                      "transposed")


@pytest.mark.parametrize("lower,upper", [(8, 2), (9, 2), (14, 2), (15, 1), (2, 9), (2, 14)])
def test_one_call_pick_by_the_side_it_sweeps(lower, upper):
    """Rows of up to 8 entries on a side are swept on the ring, longer ones by
    a cluster on DAGs this narrow, whatever the other side holds (rows of up to
    17 entries in all, for which the solve builds the level orders)."""
    n = 6000
    A = from_rows(n, lambda i: [i - 7 * j for j in range(1, lower + 1)] +
                  [i + 11 * j for j in range(1, upper + 1)], 3)
    rp, ci, av = to_dev(A)
    b, bd = vec(82, n)
    x, info, (S, F) = P.solve(rp, ci, av, bd, 0, return_factors=True)
    f, b_ = kinds(F.schedule())
    ring = (L.SCHED_SINGLE_CTA, L.SCHED_CLUSTER)
    assert (f in ring) == (lower <= 8) and (b_ in ring) == (upper <= 8)
    assert f in FEW_SMS and b_ in FEW_SMS
    ref = oracle.factor(A, 0)
    st, xo, it, *_ = oracle.gmres(n, A.rowptr, A.colind, A.val, b, oracle.PREC_ILU,
                                  (ref["rowptr"], ref["colind"], ref["val"]), 30, 1e-8,
                                  dotmode=oracle.DOT_TREE)
    assert st == oracle.OK and info.iters == it
    assert_bits_equal(x, xo, f"{lower} lower, {upper} upper")


@pytest.mark.parametrize("N,k,kind", [(128, 0, L.SCHED_SINGLE_CTA), (256, 0, L.SCHED_CLUSTER),
                                      (300, 1, L.SCHED_CLUSTER), (200, 2, L.SCHED_SINGLE_CTA)])
def test_one_call_pick_counts_rows_too(N, k, kind):
    """Levels of many short rows go to four SMs before levels of few longer
    ones with as many entries do (256^2 k = 0: 255 entries a level on 128 rows;
    200^2 k = 2: 199 on 50)."""
    A = W.conv_diff(N, 2, (20.0, 20.0))
    rp, ci, av = to_dev(A)
    b, bd = vec(83, A.n)
    x, info, (S, F) = P.solve(rp, ci, av, bd, k, maxit=2, check=False, return_factors=True)
    assert kinds(F.schedule()) == (kind, kind)


@pytest.mark.parametrize("n,hw,kind", [(160000, 2000, L.SCHED_WARP_GRID),
                                       (40000, 500, L.SCHED_WARP_CLUSTER)])
def test_one_call_pick_for_longer_rows_counts_rows_too(n, hw, kind):
    """Random bands of 9 entries a row, k = 0: 861 levels of 186 rows go to all
    SMs (an application 1.39 ms, on a cluster 1.98), 790 of 51 to a cluster
    (0.78 ms; all SMs 1.30)."""
    A = W.random_band(n, 9, hw, 77)
    rp, ci, av = to_dev(A)
    b, bd = vec(84, n)
    x, info, (S, F) = P.solve(rp, ci, av, bd, 0, maxit=2, check=False, return_factors=True)
    assert S.max_row <= 17 and kinds(F.schedule()) == (kind, kind)


def test_one_call_pick_leaves_the_ring_where_inputs_lie_far():
    """Short rows, 85 a level, but one in eight has no lower entries: level 1
    holds rows from everywhere, far behind the ring for most of their readers."""
    A = W.random_band(40000, 3, 300, 1)
    rp, ci, av = to_dev(A)
    b, bd = vec(85, A.n)
    x, info, (S, F) = P.solve(rp, ci, av, bd, 0, return_factors=True)
    assert S.max_row <= 4 and kinds(F.schedule()) == (L.SCHED_WARP_CLUSTER, L.SCHED_WARP_CLUSTER)
    ref = oracle.factor(A, 0)
    st, xo, it, *_ = oracle.gmres(A.n, A.rowptr, A.colind, A.val, b, oracle.PREC_ILU,
                                  (ref["rowptr"], ref["colind"], ref["val"]), 30, 1e-8,
                                  dotmode=oracle.DOT_TREE)
    assert st == oracle.OK and info.iters == it
    assert_bits_equal(x, xo, "far inputs")
