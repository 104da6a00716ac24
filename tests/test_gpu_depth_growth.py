"""The route a factorization takes by how the forward depth grows with the row
index, against the oracle, bit for bit: depth growing with the index (index
order, orders beside the rows), saturating (orders first, dropped again where a
factorization leaves none), a chain at the head of a shallow matrix and the
reverse (what the first rows suggest is wrong), a wide forward DAG under a deep
backward one, and sizes around the probe's least.  Level orders exist after
iluk_factor exactly where n >= 128 times the forward depth."""
import ctypes as C

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


def from_rows(rows):
    rng = np.random.default_rng(len(rows))
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    ci = np.concatenate([np.array(sorted(r), np.int32) for r in rows])
    va = rng.uniform(-0.4, 0.4, len(ci))
    va[ci == np.repeat(np.arange(len(rows)), np.diff(rp))] = 3.0
    return W.CSR(len(rows), rp, ci, va)


def head_chain(n, chain):  # rows 0 .. chain - 1 a chain, the others diagonal
    return from_rows([{i} | ({i - 1} if 0 < i < chain else set()) for i in range(n)])


def tail_chain(n, chain):
    return from_rows([{i} | ({i - 1} if i > n - chain else set()) for i in range(n)])


def backward_chain(n):  # no lower entries; each row reads the next one
    return from_rows([{i, i + 1} if i + 1 < n else {i} for i in range(n)])


CASES = [("band20000_k1", W.random_band(20000, 9, 400, 3), 1),
         ("band4095_k1", W.random_band(4095, 9, 100, 3), 1),
         ("band4096_k2", W.random_band(4096, 9, 100, 3), 2),
         ("band40000_k0", W.random_band(40000, 3, 9000, 5), 0),
         ("grid2d_150_k1", W.conv_diff(150, 2, (20.0, 20.0)), 1),
         ("grid3d_28_k0", W.conv_diff(28, 3, (50.0, 50.0, 50.0)), 0),
         ("poisson27_28_k1", W.poisson27(28), 1),
         ("head_chain_wide", head_chain(40000, 300), 0),
         ("head_chain_narrow", head_chain(40000, 4000), 1),
         ("tail_chain", tail_chain(20000, 3000), 1),
         ("tridiagonal", from_rows([{j for j in (i - 1, i, i + 1) if 0 <= j < 5000}
                                    for i in range(5000)]), 0),
         ("diagonal", head_chain(20000, 0), 0),
         ("backward_chain", backward_chain(6000), 0)]


def forward_depth(ref, n):
    d = np.zeros(n, np.int64)
    rp, ci = ref["rowptr"], ref["colind"]
    for i in range(n):
        lo = ci[rp[i]:rp[i + 1]]
        lo = lo[lo < i]
        d[i] = 1 + (d[lo].max() if len(lo) else 0)
    return int(d.max())


@pytest.mark.parametrize("name,A,k", CASES, ids=[c[0] for c in CASES])
def test_routes_bit_exact(name, A, k):
    rp, ci, av = to_dev(A)
    ref = oracle.factor(A, k)
    depth = forward_depth(ref, A.n)
    S, F = P.factor(rp, ci, av, k)
    view = L.SymView()
    assert L.load().iluk_sym_query(S.h, C.byref(view)) == 0
    assert view.depth_lower == (depth if A.n >= 128 * depth else -1)
    assert_bits_equal(F.values(), ref["val"], f"{name}: factor")
    b, bd = vec(31, A.n)
    y = oracle.apply(A.n, ref["rowptr"], ref["colind"], ref["val"], b)
    assert_bits_equal(F.apply(bd), y, f"{name}: apply")
    S2 = P.symbolic(rp, ci, k)
    F2 = P.numeric(S2, av)
    assert_bits_equal(F2.values(), ref["val"], f"{name}: numeric")
    assert S2.depth()[0] == depth
    F2.refactor(av)
    assert_bits_equal(F2.values(), ref["val"], f"{name}: refactor")
    st, xo, it, rel, cyc = oracle.gmres(A.n, A.rowptr, A.colind, A.val, b, oracle.PREC_ILU,
                                        (ref["rowptr"], ref["colind"], ref["val"]), 20, 1e-10,
                                        dotmode=oracle.DOT_TREE)
    x, info = P.solve(rp, ci, av, bd, k=k, restart=20, rtol=1e-10)
    assert (info.iters, info.cycles) == (it, cyc)
    assert_bits_equal(x, xo, f"{name}: solve")


def test_zero_pivot_beside_the_orders():
    A = W.random_band(20000, 9, 400, 3)
    rp, ci, av = to_dev(A)
    zero = torch.zeros_like(av)
    for call in (lambda: P.factor(rp, ci, zero, 1), lambda: P.numeric(P.symbolic(rp, ci, 1), zero)):
        with pytest.raises(P.IlukError) as e:
            call()
        assert e.value.status == L.EZEROPIVOT and e.value.row == 0
