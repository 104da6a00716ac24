"""The batched sweeps on the packed copy of the factors against the oracle, bit
for bit, where they can go wrong: chains one shorter than, as long as and longer
than the packed part, levels at the width from which the copy is made and one
row narrower, and levels that fill a warp exactly or by one row more."""
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


def blocks(count, size):
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


@pytest.mark.parametrize("width", [256, 512, 1024])
@pytest.mark.parametrize("count,size", [(3, 8), (4, 6), (4, 7), (4, 8), (32, 7), (33, 9), (70, 20)])
def test_packed_sweeps_bit_exact(count, size, width):
    A = blocks(count, size)
    rp, ci, av = to_dev(A)
    S = P.symbolic(rp, ci, 0)
    items, mats = [], []
    for scale in (1.0, -2.5):
        b = torch.linspace(-1.0, scale, A.n, dtype=torch.float64, device="cuda")
        items.append((S, av * scale, b, torch.zeros_like(b)))
        mats.append(W.CSR(A.n, A.rowptr, A.colind, A.val * scale))
    B = P.BatchSolve(items, restart=30, rtol=1e-8)
    B.set_schedule(width, True)
    B.solve()
    for M, (_, _, b, x), r in zip(mats, items, B.results()):
        F = oracle.factor(M, 0)
        st, xo, it, rel, cyc = oracle.gmres(M.n, M.rowptr, M.colind, M.val, b.cpu().numpy(),
                                            oracle.PREC_ILU, (F["rowptr"], F["colind"], F["val"]),
                                            30, 1e-8, dotmode=oracle.DOT_TREE)
        assert r.status == st == 0 and (r.iters, r.cycles) == (it, cyc)
        assert_bits_equal(x, xo, f"{count} x {size}")
