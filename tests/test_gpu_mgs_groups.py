"""The groups in which the one-launch Gram-Schmidt step adds its products,
against the oracle (fixed-tree inner products), bit for bit: rows of partials
around a group, around pairs of groups, around the sizes where the group
changes, with the last row full, holding one element and all but one, and the
most rows the shared memory holds and one more (one inner product a launch)."""
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


def bidiagonal(n):
    rp = np.concatenate([[0, 1], 1 + 2 * np.arange(1, n)]).astype(np.int64)
    ci = np.zeros(2 * n - 1, np.int32)
    va = np.zeros(2 * n - 1)
    i = np.arange(n)
    ci[rp[1:] - 1], va[rp[1:] - 1] = i, 2.0 + (i % 7) / 8.0
    ci[1::2], va[1::2] = i[:-1], -0.75 - (i[1:] % 3) / 4.0
    return W.CSR(n, rp, ci, va)


@pytest.mark.parametrize("last", [1, 4095, 4096])
@pytest.mark.parametrize("rows", [1, 3, 4, 5, 8, 9, 12, 13, 63, 64, 65, 72, 73, 80, 81, 221, 222])
def test_groups_bit_exact(rows, last):
    n = (rows - 1) * 4096 + last
    A = bidiagonal(n) if n > 1 else W.CSR(1, np.array([0, 1]), np.zeros(1, np.int32), np.ones(1))
    rp, ci, av = to_dev(A)
    b, bd = vec(rows, n)
    args = (5, 1e-13, 6)
    st, xo, it, rel, cyc = oracle.gmres(A.n, A.rowptr, A.colind, A.val, b, oracle.PREC_NONE, None,
                                        *args, dotmode=oracle.DOT_TREE)
    x, info = P.gmres(rp, ci, av, bd, None, restart=5, rtol=1e-13, maxit=6, check=False)
    assert (info.status, info.iters, info.cycles) == (st, it, cyc)
    assert bits([info.relres])[0] == bits([rel])[0]
    assert_bits_equal(x, xo, f"rows {rows}, last {last}")
