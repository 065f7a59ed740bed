"""Contexts of several host threads, each on its own stream: a thread's calls must
not change what another thread's launches are allowed (a kernel's shared-memory
limit is the kernel's, not the launch's)."""
import threading

import numpy as np
import pytest

from oracle import quadrature
from paper_1006_3340_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1006_3340_gb300 import lll

    lll.load()
    return torch, lll


def _signed(x, W):
    """A rule of the same length with one negative weight (no shorter rule stands for it)."""
    j = int(np.argmin(np.abs(x)))
    W = W.copy()
    W[j] *= -0.5
    return x, W


def _together(torch, jobs):
    """Run the jobs on a thread and a stream each, started together; the exceptions they raised."""
    gate, errors = threading.Barrier(len(jobs)), []

    def body(job):
        torch.cuda.set_device(0)
        stream = torch.cuda.Stream()
        gate.wait()
        try:
            job(stream.cuda_stream)
        except Exception as e:  # reported by the caller
            errors.append(e)

    threads = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


def test_contexts_with_long_rules_are_built_from_two_threads(env):
    torch, lll = env

    def build(Q):
        wl = workloads.tiny(N=3, s=1, Q=Q)
        x, W = _signed(*quadrature.rule_for(wl))

        def job(stream):
            for _ in range(3000):
                lll.LevyLibor(wl, x, W, stream=stream).close()

        return job

    assert not _together(torch, [build(96), build(128)])
