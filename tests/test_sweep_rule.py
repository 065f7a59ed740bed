"""The shorter rule of the sweeps (lll_sweep_rule) against the rule as given, in
FP64 on the host: the state-dependent part of the compensator,
    A_i - C_i = sum_j W_j / x_j^2 (e^{lambda_i x_j} - 1)(P(x_j) - 1),
    P = prod_{l > i} (1 - w_l + w_l e^{lambda_l x}),
agrees to 2^-28 of its terms for every state, w_l anywhere in [0, 1], where the
volatilities' sums stay within [lo, hi].  The bound is the rule's own criterion
(a relative error of the generating function), and P a convex combination of
exponentials, so nothing else enters but FP64 rounding, which the cancellation
of E and of P - 1 next to 0 lets grow to 1e-12 of the terms.
"""
import numpy as np
import pytest

from oracle import quadrature
from paper_1006_3340_gb300 import build as libbuild

TOL = 2.0 ** -28 + 1e-11


@pytest.fixture(scope="module")
def lll():
    libbuild.build()
    from paper_1006_3340_gb300 import lll as mod

    mod.load()
    return mod


def _dependent(x, W, lam, w):
    """A_i - C_i and the sum of its terms' absolute values (over nodes and subsets'
    signs: |e^{lambda x} - 1| |P - 1| bounded by the same with |lambda|, |x|)."""
    E = np.expm1(np.multiply.outer(lam, x))
    P = np.prod(1.0 + w[1:, None] * E[1:], axis=0)
    return np.sum(W / x ** 2 * E[0] * (P - 1.0))


def _mass(x, W, lam, w):
    a = np.abs(lam)
    E = np.abs(np.expm1(np.multiply.outer(a, np.abs(x))))
    P = np.prod(1.0 + w[1:, None] * E[1:], axis=0)
    return np.sum(W / x ** 2 * E[0] * (P - 1.0))


@pytest.mark.parametrize("alpha,beta,dbar,a,Q", [(18.0, -4.0, 1.0, 1.5, 32), (12.0, -3.0, 0.8, 1.5, 64),
                                                 (10.0, -2.5, 1.2, 1.5, 96), (1.5, 0.0, 1.5, 30.0, 96),
                                                 (9.0, -2.0, 1.0, 1.5, 8), (25.0, 3.0, 1.0, 1.5, 128)])
@pytest.mark.parametrize("n", [1, 9, 39])
@pytest.mark.parametrize("signs", ["positive", "mixed"])
def test_shorter_rule_gives_the_given_rules_drift(lll, alpha, beta, dbar, a, Q, n, signs):
    x, W = quadrature.gauss_rule(alpha, beta, dbar, a, Q)
    rng = np.random.default_rng(Q + n)
    lam = rng.uniform(0.02, 0.2, n + 1)
    if a > 10:
        lam *= 1.4 / lam.sum()  # the heavy-tailed rule reaches to |x| = 30
    if signs == "mixed":
        lam *= rng.choice([-1.0, 1.0], n + 1)
    lo, hi = lam[lam < 0].sum(), lam[lam > 0].sum()
    xr, wr, padded = lll.lll_sweep_rule(x, W, lo, hi)
    if len(xr) == 0:
        assert padded >= Q
        return
    assert len(xr) <= padded <= min(Q, 32) and np.all(wr > 0)
    assert np.sum(wr / np.abs(xr)) <= np.sum(W / np.abs(x)) * (1 + 1e-12)
    for w in [np.zeros(n + 1), np.ones(n + 1), np.full(n + 1, 0.01)] + [rng.uniform(0, 1, n + 1) for _ in range(5)] + \
            [rng.uniform(0, 0.05, n + 1) for _ in range(5)]:
        err = abs(_dependent(xr, wr, lam, w) - _dependent(x, W, lam, w))
        assert err <= TOL * _mass(x, W, lam, w), (len(xr), err)


def test_short_for_ordinary_rules_and_none_where_it_does_not_stand(lll):
    x, W = quadrature.gauss_rule(12.0, -3.0, 0.8, 1.5, 64)
    assert 0 < len(lll.lll_sweep_rule(x, W, 0.0, 4.3)[0]) <= 8
    # one node of the measure: the rule is that node
    one = lll.lll_sweep_rule([0.5], [1.0], 0.0, 2.0)
    assert len(one[0]) == 1 and abs(one[0][0] - 0.5) < 1e-14 and abs(one[1][0] - 1.0) < 1e-14 and one[2] == 4
    # no Gauss rule of a signed measure; a node next to 0; sums beyond any short rule; overflow
    V = W.copy()
    V[5] = -V[5]
    y = x.copy()
    y[np.argmin(np.abs(x))] = 3e-5
    for args in ((x, V, 0.0, 4.3), (y, W, 0.0, 4.3), (x, W, 0.0, 1e3), (x, W, -1e300, 1e300)):
        xr, wr, padded = lll.lll_sweep_rule(*args)
        assert len(xr) == 0 and padded == 64
    with pytest.raises(lll.LLLError):
        lll.lll_sweep_rule(x, W, 1.0, 2.0)
