"""The one-launch Gram-Schmidt step of GMRES against the oracle (fixed-tree
inner products), bit for bit, at its edges: fewer elements than partials, one
row of partials and its neighbours, chunk boundaries (four rows), and the most
elements the CTAs hold and one more (one inner product a launch)."""
import numpy as np
import pytest
import torch

import oracle
import paper_0803_0048_gb300 as P
from paper_0803_0048_gb300 import workloads as W

from gpu_helpers import assert_bits_equal, bits, to_dev, vec

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def tridiagonal(n):
    i = np.arange(n)
    cols = np.stack([i - 1, i, i + 1], axis=1)
    vals = np.tile([-1.0, 2.5, -0.75], (n, 1)) * (1.0 + (i % 5)[:, None] / 8.0)
    ok = (cols >= 0) & (cols < n)
    rp = np.zeros(n + 1, dtype=np.int64)
    rp[1:] = np.cumsum(ok.sum(axis=1))
    return W.CSR(n, rp, cols[ok].astype(np.int32), vals[ok])


@pytest.mark.parametrize("n", [1, 2, 31, 33, 4095, 4096, 4097, 8200, 35 * 4096, 36 * 4096 + 5, 216 * 4096,
                               39 * 4096 + 4000, 216 * 4096 + 1])
@pytest.mark.parametrize("restart", [3, 30])
def test_gmres_edges_bit_exact(n, restart):
    A = tridiagonal(n)
    rp, ci, av = to_dev(A)
    b, bd = vec(n + restart, n)
    maxit = 7 if n > 100000 else 12
    st, xo, it, rel, cyc = oracle.gmres(A.n, A.rowptr, A.colind, A.val, b, oracle.PREC_NONE, None,
                                        restart, 1e-12, maxit, dotmode=oracle.DOT_TREE)
    x, info = P.gmres(rp, ci, av, bd, None, restart=restart, rtol=1e-12, maxit=maxit, check=False)
    assert (info.status, info.iters, info.cycles) == (st, it, cyc)
    assert bits([info.relres])[0] == bits([rel])[0]
    assert_bits_equal(x, xo, f"n = {n}")


def test_gmres_breakdown_and_non_finite():
    # A = 2 I: the first step's norm is exactly zero
    n = 5000
    A = W.CSR(n, np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32), np.full(n, 2.0))
    rp, ci, av = to_dev(A)
    b, bd = vec(5, n)
    x, info = P.gmres(rp, ci, av, bd, None, restart=10, rtol=1e-12)
    st, xo, it, rel, cyc = oracle.gmres(A.n, A.rowptr, A.colind, A.val, b, oracle.PREC_NONE, None,
                                        10, 1e-12, dotmode=oracle.DOT_TREE)
    assert (info.status, info.iters, info.cycles) == (st, it, cyc)
    assert_bits_equal(x, xo, "x")
    # a NaN in b: the norms are NaN, nothing hangs, no convergence
    bd[17] = float("nan")
    x, info = P.gmres(rp, ci, av, bd, None, restart=5, rtol=1e-12, maxit=6, check=False)
    assert info.status != 0
