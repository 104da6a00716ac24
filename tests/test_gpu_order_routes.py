"""Whether the level orders are built before the rows or beside them follows from
the DAG's shape: told by the profile (orders beside the rows count as overlapped),
for the two calls and the one-call factorization, with the oracle's values."""
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


def grid(nx, ny):
    """5-point stencil, x fastest, on nx * ny points."""
    i = np.arange(nx * ny)
    x, y = i % nx, i // nx
    cols = np.stack([np.where(y > 0, i - nx, -1), np.where(x > 0, i - 1, -1), i,
                     np.where(x < nx - 1, i + 1, -1), np.where(y < ny - 1, i + nx, -1)], 1)
    keep = cols >= 0
    rp = np.zeros(len(i) + 1, np.int64)
    rp[1:] = np.cumsum(keep.sum(1))
    val = np.random.default_rng(nx).uniform(-1, 1, cols.shape)
    val[:, 2] = 5.0
    return W.CSR(len(i), rp, cols[keep].astype(np.int32), val[keep])


FIRST, BESIDE = "depth", "overlapped"
# (pattern, k, the two calls' route)
CASES = [("grid256x256", grid(256, 256), 0, FIRST), ("grid1024x64", grid(1024, 64), 0, FIRST),
         ("grid128x512", grid(128, 512), 0, FIRST), ("grid64x1024", grid(64, 1024), 0, BESIDE),
         ("grid30x1500", grid(30, 1500), 0, BESIDE), ("grid3d_64_k0",
                                                      W.conv_diff(64, 3, (5.0, 5.0, 5.0)), 0, FIRST),
         ("grid3d_32_k1", W.conv_diff(32, 3, (5.0, 5.0, 5.0)), 1, FIRST),
         ("grid3d_20_k2", W.conv_diff(20, 3, (5.0, 5.0, 5.0)), 2, BESIDE),
         ("grid141_few_rows", grid(141, 141), 0, BESIDE), ("grid142", grid(142, 142), 0, FIRST),
         ("poisson27_28_k0", W.poisson27(28), 0, FIRST),
         ("band160k_k0", W.random_band(160000, 9, 2000, 3), 0, BESIDE),
         ("band40k_4_k0", W.random_band(40000, 4, 1000, 3), 0, BESIDE),
         ("band60k_k1", W.random_band(60000, 9, 300, 3), 1, BESIDE)]


@pytest.mark.parametrize("name,A,k,route", CASES, ids=[c[0] for c in CASES])
def test_orders_first_or_beside(name, A, k, route):
    rp, ci, av = to_dev(A)
    ref = oracle.factor(A, k)
    S = P.symbolic(rp, ci, k)
    P.prof_enable(True)
    F = P.numeric(S, av)
    prof = P.prof_read()
    P.prof_enable(False)
    assert (prof.get(BESIDE, (0, 0))[1] > 0) == (route == BESIDE), prof
    assert_bits_equal(F.values(), ref["val"], name)
    _, F2 = P.factor(rp, ci, av, k)
    assert_bits_equal(F2.values(), ref["val"], name + " in one call")
