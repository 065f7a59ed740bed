"""Contexts of several host threads, each on its own stream: a thread's calls must
not change what another thread's launches are allowed (a kernel's shared-memory
limit is the kernel's, not the launch's)."""
import dataclasses
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


@pytest.mark.parametrize("scheme,setup,shapes", [
    ("full", lambda s: s.set_launch(64, 0, 0, 1, 1), (3, 40)),        # one path a thread, the rule as given
    ("full", lambda s: s.set_launch(64, 0, 0, 1, 4), (3, 40)),        # lane groups
    ("picard", lambda s: s.set_mapping("tenor", 8), (3, 40)),
    ("picard", lambda s: s.set_mapping("step"), (3, 120)),
    ("expand1", lambda s: None, (3, 24))])
def test_simulations_of_two_sizes_from_two_threads(env, scheme, setup, shapes):
    """The two models' launches need different amounts of shared memory, one more than
    the 48 KB that a kernel has without asking."""
    torch, lll = env
    want, jobs, got = {}, [], {}
    for N in shapes:
        wl = workloads.tiny(N=N, s=1, Q=128 if N == 120 else 64, paths=64)
        wl = dataclasses.replace(wl, lam=np.full_like(wl.lam, 0.02), L0=np.full(N, 0.03),
                                 strikes=np.tile(wl.strikes[:1], (wl.n, 20 if N < 100 else 5)))
        rule = _signed(*quadrature.rule_for(wl))

        def job(stream, N=N, wl=wl, rule=rule, rounds=3000):
            sim = lll.LevyLibor(wl, *rule, stream=stream)
            try:
                setup(sim)
                for _ in range(rounds):
                    sim.simulate(scheme)
                got[N] = sim.prices()[0]
            finally:
                sim.close()

        job(0, rounds=1)
        want[N] = got[N]
        jobs.append(job)
    assert not _together(torch, jobs)
    for N in shapes:
        assert np.array_equal(got[N], want[N])
