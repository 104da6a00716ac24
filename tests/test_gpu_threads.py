"""Threads on streams of their own, each with patterns that need another amount
of shared memory in the same kernels: every call returns OK and the right bits."""
import threading

import numpy as np
import pytest
import torch

import paper_0803_0048_gb300 as P
from paper_0803_0048_gb300 import workloads as W

from gpu_helpers import assert_bits_equal, to_dev, vec

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def run_threads(bodies):
    errors = []

    def guarded(body):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                body()
                torch.cuda.current_stream().synchronize()
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=guarded, args=(b,)) for b in bodies]
    torch.cuda.synchronize()
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[:2]


def dense_blocks(count, size):
    rng = np.random.default_rng(size)
    n = count * size
    ci = np.repeat(np.arange(count), size * size) * size + np.tile(np.arange(size), n)
    va = rng.uniform(-1, 1, n * size)
    va[np.arange(n) * size + np.tile(np.arange(size), count)] = size + 1.0
    return W.CSR(n, np.arange(n + 1, dtype=np.int64) * size, ci.astype(np.int32), va)


def test_refactor_in_threads():
    """Rows of 60 entries beside rows of 2 and 7, on update plans."""
    mats = [dense_blocks(60, 60), dense_blocks(200, 2), W.conv_diff(24, 3, (50.0, 50.0, 50.0))]
    made = []
    for A in mats:
        rp, ci, av = to_dev(A)
        F = P.numeric(P.symbolic(rp, ci, 0), av)
        made.append((F, av, F.values()))

    def body(F, av):
        def go():
            for _ in range(400):
                F.refactor(av)
        return go

    run_threads([body(F, av) for F, av, _ in made])
    for F, _, want in made:
        assert_bits_equal(F.values(), want, "after the threads")


def test_symbolic_in_threads():
    """Windows of 5, 201 and up to 7,999 columns."""
    mats = [W.random_band(3000, 2, 2, 1), W.random_band(3000, 9, 100, 2),
            W.random_sparse(4000, 0.001, 3)]
    dev = [to_dev(A) for A in mats]
    want = [[t.cpu() for t in P.symbolic(rp, ci, 2).pattern()] for rp, ci, _ in dev]

    def body(rp, ci, w):
        def go():
            for _ in range(150):
                S = P.symbolic(rp, ci, 2)
            assert all(torch.equal(a.cpu(), b) for a, b in zip(S.pattern(), w))
        return go

    run_threads([body(rp, ci, w) for (rp, ci, _), w in zip(dev, want)])


def test_gmres_in_threads():
    """Vectors of one row of partial sums beside vectors of sixteen."""
    mats = [W.conv_diff(60, 2, (20.0, 20.0)), W.conv_diff(250, 2, (20.0, 20.0))]
    made = []
    for A in mats:
        rp, ci, av = to_dev(A)
        _, b = vec(5, A.n)
        x, info = P.gmres(rp, ci, av, b, None, restart=20, rtol=1e-30, maxit=60, check=False)
        made.append((rp, ci, av, b, x))

    def body(rp, ci, av, b, want):
        def go():
            for _ in range(25):
                x, _ = P.gmres(rp, ci, av, b, None, restart=20, rtol=1e-30, maxit=60, check=False)
            assert_bits_equal(x, want, "gmres")
        return go

    run_threads([body(*m) for m in made])
