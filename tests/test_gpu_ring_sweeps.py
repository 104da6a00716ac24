"""The lockstep sweeps on the shared-memory ring (SINGLE_CTA and CLUSTER)
against the oracle, bit for bit, at the sizes where they can go wrong: one
row, one chunk of 32 rows and its edges, rows of exactly the window sizes and
one beyond (2 + 2, 4 + 4, and longer ones that run warp-per-row),
levels wider than the warps, and orders long enough that inputs lie beyond the
ring or are overwritten in it (more than 8,192 slots back)."""
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


def from_lower(n, lower, seed):
    """Rows i with lower columns lower(i) (and their mirror), dominant."""
    rng = np.random.default_rng(seed)
    rows = [[] for _ in range(n)]
    for i in range(n):
        for j in sorted(set(lower(i))):
            rows[i].append(j)
            rows[j].append(i)
    rp, ci, va = [0], [], []
    for i in range(n):
        cols = sorted(set(rows[i]) | {i})
        ci += cols
        va += [float(len(cols)) + 1.0 if c == i else rng.uniform(-1, 1) for c in cols]
        rp.append(len(ci))
    return W.CSR(n, np.array(rp, np.int64), np.array(ci, np.int32), np.array(va))


def entries(w):
    """Every row reads the w rows before it (a chain), w entries a row."""
    return lambda i: [j for j in range(i - w, i) if j >= 0]


CASES = [("n1", from_lower(1, entries(0), 1), 0),
         ("n31_diag", from_lower(31, entries(0), 2), 0),
         ("n33_diag", from_lower(33, entries(0), 3), 0)]
CASES += [(f"chain_w{w}", from_lower(97, entries(w), 10 + w), 0) for w in (1, 4, 5, 8, 9, 16, 17)]
CASES += [("wide_levels", from_lower(2500, lambda i: [i - 1250] if i >= 1250 else [], 4), 0),
          # 20,000 independent rows, then rows that read across them: slots
          # far behind the ring, and a few close by
          ("far_back", from_lower(20600, lambda i: [] if i < 20000 else
                                  [(37 * i) % 20000, (11 * i) % 300, i - 1], 5), 0),
          # a chain whose rows also read row 0's neighbourhood from 9,000 rows on
          ("overwritten", from_lower(9400, lambda i: [i - 1] * (i > 0) +
                                     ([i - 9000] if i >= 9000 else []), 6), 0),
          ("convdiff2d_40_k2", W.conv_diff(40, 2, (20.0, 20.0)), 2),
          ("convdiff3d_20_k1", W.conv_diff(20, 3, (50.0, 50.0, 50.0)), 1),
          ("poisson27_9_k0", W.poisson27(9), 0)]


@pytest.mark.parametrize("name,A,k", CASES, ids=[c[0] for c in CASES])
@pytest.mark.parametrize("sched", [L.SCHED_SINGLE_CTA, L.SCHED_CLUSTER,
                                   L.SCHED_SINGLE_CTA | (L.SCHED_CLUSTER << 8)])
def test_ring_sweeps_bit_exact(name, A, k, sched):
    rp, ci, av = to_dev(A)
    F = P.numeric(P.symbolic(rp, ci, k), av)
    ref = oracle.factor(A, k)
    trp, tci, tv = oracle.transpose(A.n, ref["rowptr"], ref["colind"], ref["val"])
    for rep in range(2):
        p, pd = vec(40 + rep, A.n)
        assert_bits_equal(F.apply(pd, sched=sched),
                          oracle.apply(A.n, ref["rowptr"], ref["colind"], ref["val"], p), name)
        assert_bits_equal(F.apply(pd, transpose=True, sched=sched),
                          oracle.apply_t(A.n, trp, tci, tv, p), name + " transposed")
    assert F.status() == L.OK


def test_ring_sweep_in_a_capture():
    """A plan is not built inside a capture: a first use there runs as the
    warp-per-row grid; with the plan made before, the captured sweep replays
    on new values of the same pattern."""
    A = W.conv_diff(24, 2, (20.0, 20.0))
    rp, ci, av = to_dev(A)
    ref = oracle.factor(A, 2)
    for planned in (False, True):
        F = P.numeric(P.symbolic(rp, ci, 2), av)
        p, pd = vec(7, A.n)
        y = torch.empty_like(pd)
        if planned:
            F.apply(pd, out=y, sched=L.SCHED_SINGLE_CTA)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            F.apply(pd, out=y, sched=L.SCHED_SINGLE_CTA)
        for scale in (1.0, 1.25):
            F.refactor(av * scale)
            r = oracle.factor(W.CSR(A.n, A.rowptr, A.colind, A.val * scale), 2)
            g.replay()
            torch.cuda.synchronize()
            assert_bits_equal(y, oracle.apply(A.n, r["rowptr"], r["colind"], r["val"], p),
                              f"planned {planned} scale {scale}")
    assert ref["val"].size
