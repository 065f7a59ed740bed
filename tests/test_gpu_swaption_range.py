"""Swaptions whose values leave FP32's exponents: the payoffs of the time-blocked
and step-parallel kernels on a rule with a shorter equivalent, against the same
payoff in FP64 on the paths that the library itself recorded.

Tolerance: a recorded log-rate is the kernel's FP32 offset plus log L(0), rounded
once (2^-24 of at most 4), and the kernel forms L = L(0) e^offset in FP32, so each
factor 1 + delta L of a path agrees to 2^-20 and a product of n of them, or their
sum, to n 2^-20; a payoff (X - K S)^+ to that of its terms."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as ora
from oracle import quadrature
from paper_1006_3340_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lll():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1006_3340_gb300 import lll as mod

    mod.load()
    return mod


def _expected(wl, z):
    """Mean and standard error of the swaption payoffs, and the mean of their terms."""
    P, n, d = len(z), wl.n, wl.delta
    mean, se, mass = (np.zeros(wl.strikes.shape) for _ in range(3))
    BN = ora.discount_terminal(wl)
    for m in range(1, n + 1):
        f = 1.0 + d * np.exp(z[:, m - 1, m - 1:].astype(np.float64))      # L_m .. L_n
        tail = np.cumprod(f[:, :0:-1], axis=1)                              # prod over l > m, then fewer
        S = 1.0 + tail.sum(axis=1)
        X = np.prod(f, axis=1) - 1.0
        for q, K in enumerate(wl.strikes[m - 1]):
            v = BN * np.maximum(X - float(np.float32(K)) * d * S, 0.0)
            mean[m - 1, q], se[m - 1, q] = v.mean(), v.std(ddof=1) / np.sqrt(P)
            mass[m - 1, q] = BN * (X + abs(K) * d * S).mean()
    return mean, se, mass


MODELS = {  # forward rate, tenors, strikes
    "squares beyond": (1.5, 52, [0.0, 1.0, 1.5, 1.6]),
    "products beyond": (1.5, 98, [0.0, 1.0, 1.5, 1.6]),
    "strike beyond": (0.03, 20, [0.03, 5e3, -5e3, -1e19]),
    "within": (0.03, 20, [0.0, 0.03, -1.0, 999.0]),
}


@pytest.mark.parametrize("model", MODELS)
@pytest.mark.parametrize("scheme,launch,mapping", [("full", (32, 0, 0, 1, 1), "path"), ("full", (128, 0, 0, 2, 1), "path"),
                                                   ("picard", (64, 0, 0, 1, 1), "path"), ("picard", (64, 0, 0, 2, 1), "path"),
                                                   ("picard", (128, 0, 0, 1, 1), "step"), ("full", (0, 0, 0, 0, 0), "path")])
def test_swaptions_of_any_size(lll, model, scheme, launch, mapping):
    rate, N, K = MODELS[model]
    wl = workloads.tiny(N=N, s=2, Q=64, paths=301)
    wl = dataclasses.replace(wl, delta=1.0, L0=np.full(N, rate), lam=np.full_like(wl.lam, 0.02), strikes=np.tile(K, (wl.n, 1)))
    x, W = quadrature.rule_for(wl)
    assert len(lll.lll_sweep_rule(x, W, 0.0, 0.02 * wl.n)[0]) > 0
    sim = lll.LevyLibor(wl, x, W)
    try:
        sim.set_product("swaption")
        sim.set_launch(*launch)
        sim.set_mapping(mapping)
        sim.simulate(scheme, snapshots=wl.paths)
        z = sim.paths(0, wl.paths)
        p, se = sim.prices()
    finally:
        sim.close()
    want, want_se, mass = _expected(wl, z)
    tol = wl.n * 2.0 ** -20
    assert np.all(np.isfinite(p)) and np.all(np.isfinite(se))
    assert np.all(np.abs(p - want) <= tol * mass)
    assert np.all(np.abs(se - want_se) <= 4 * tol * mass)
