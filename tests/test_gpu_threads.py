"""Threads on streams of their own, each with patterns that need another amount
of shared memory in the same kernels: every call returns OK and the right bits."""
import threading

import pytest
import torch

import paper_0803_0048_gb300 as P
from paper_0803_0048_gb300 import workloads as W

from gpu_helpers import to_dev

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
