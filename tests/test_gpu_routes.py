"""Kernels that a default launch of the ordinary workloads no longer reaches, path by
path against the FP64 oracle on the rule as given: the step-parallel kernels at
every node count, the one-lane and step-parallel kernels of rules without a shorter
equivalent, more strikes than threads, two paths a thread with swaptions, and
volatilities of both signs.  Bars as in test_gpu_parity.py (FP32 path state: 1e-5
on rates, 1e-7 on prices)."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as ora
from oracle import quadrature
from paper_1006_3340_gb300 import workloads
from test_gpu_swaption_range import _expected

pytestmark = pytest.mark.gpu
SCHEMES = {"full": ora.FULL, "picard": ora.PICARD}
ONE_LANE = (128, 0, 0, 1, 1)


@pytest.fixture(scope="module")
def lll():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1006_3340_gb300 import lll as mod

    mod.load()
    return mod


def _check(lll, wl, x, W, scheme, paths, launch=None, mapping="path", product="caplet"):
    sim = lll.LevyLibor(wl, x, W)
    try:
        if launch:
            sim.set_launch(*launch)
        sim.set_mapping(mapping)
        sim.set_product(product)
        sim.simulate(scheme, paths=paths, snapshots=paths)
        z = sim.paths(0, paths).astype(np.float64)
        p, _ = sim.prices()
    finally:
        sim.close()
    ref = ora.simulate(ora.OracleModel(wl, x, W), SCHEMES[scheme], npaths=paths, want_snap=True)
    mask = ~np.isnan(ref["snap"])
    assert np.array_equal(mask, ~np.isnan(z))
    assert np.abs(np.expm1(z[mask] - ref["snap"][mask])).max() <= 1e-5
    want = ref["price"] if product == "caplet" else ora.swaption_prices(wl, ref["snap"], wl.strikes)
    assert np.abs(p - want).max() <= 1e-7


def _flat(N, s, Q, level, strikes=None):
    wl = workloads.tiny(N=N, s=s, Q=Q)
    wl = dataclasses.replace(wl, lam=np.full_like(wl.lam, level), L0=np.full(N, 0.03))
    return wl if strikes is None else dataclasses.replace(wl, strikes=np.tile(strikes, (wl.n, 1)))


def _signed(wl):
    """The workload's rule with one node's weight split into 1.5 and -0.5 of it: the
    same measure, which no shorter rule stands for."""
    x, W = quadrature.rule_for(wl)
    j = int(np.argmin(np.abs(x - 0.3)))
    x, W = np.append(x[1:], x[j]), np.append(W[1:], -0.5 * W[j])
    W[j - 1] *= 1.5
    return x, W


STEP_SHAPES = [(2, 1, 0.12, 4), (5, 9, 0.12, 4), (41, 3, 0.05, 8), (34, 5, 0.15, 12), (40, 2, 0.24, 16), (60, 3, 0.27, 20),
               (70, 2, 0.28, 24)]


@pytest.mark.parametrize("N,s,level,padded", STEP_SHAPES)
def test_step_kernels_of_shorter_rules(lll, N, s, level, padded):
    wl = _flat(N, s, 64, level)
    x, W = quadrature.rule_for(wl)
    assert lll.lll_sweep_rule(x, W, 0.0, level * wl.n)[2] == padded
    _check(lll, wl, x, W, "picard", 200, ONE_LANE, "step")


@pytest.mark.parametrize("N,s,level,padded", STEP_SHAPES)
def test_step_swaptions_of_shorter_rules(lll, N, s, level, padded):
    """Prices against the payoffs, in FP64, of the rates that the library recorded: a
    factor 1 + delta L agrees to 2^-20 (test_gpu_swaption_range.py), n of them to n 2^-20
    of the payoff's terms."""
    wl = _flat(N, s, 64, level)
    x, W = quadrature.rule_for(wl)
    sim = lll.LevyLibor(wl, x, W)
    try:
        sim.set_launch(*ONE_LANE)
        sim.set_mapping("step")
        sim.set_product("swaption")
        sim.simulate("picard", paths=200, snapshots=200)
        z = sim.paths(0, 200).astype(np.float64)
        p, _ = sim.prices()
    finally:
        sim.close()
    want, _, terms = _expected(wl, z)
    assert np.all(np.abs(p - want) <= wl.n * 2.0 ** -20 * terms)


@pytest.mark.parametrize("launch", [ONE_LANE, (0, 0, 0, 0, 0)])
def test_step_kernels_of_the_longest_shorter_rule(lll, launch):
    wl = workloads.paper_example()
    x, W = quadrature.rule_for(wl)
    assert lll.lll_sweep_rule(x, W, 0.0, wl.lam.sum(1).max())[2] == 32
    _check(lll, wl, x, W, "picard", 300, launch, "step")


@pytest.mark.parametrize("Q", [9, 16, 32, 64, 96, 128])
@pytest.mark.parametrize("scheme,mapping", [("full", "path"), ("picard", "path"), ("picard", "step")])
@pytest.mark.parametrize("product", ["caplet", "swaption"])
def test_rules_swept_as_given(lll, Q, scheme, mapping, product):
    wl = _flat(12, 3, Q - 1, 0.15)
    x, W = _signed(wl)
    assert len(x) == Q - 1 and len(lll.lll_sweep_rule(x, W, 0.0, 0.15 * wl.n)[0]) == 0
    _check(lll, wl, x, W, scheme, 333, None, mapping, product)


@pytest.mark.parametrize("strikes", [32, 33, 64])
@pytest.mark.parametrize("ppt", [1, 2])
@pytest.mark.parametrize("product", ["caplet", "swaption"])
def test_more_strikes_than_threads(lll, strikes, ppt, product):
    wl = _flat(9, 3, 64, 0.12, np.linspace(0.01, 0.06, strikes))
    x, W = quadrature.rule_for(wl)
    _check(lll, wl, x, W, "full", 99, (32, 0, 0, ppt, 1), product=product)


@pytest.mark.parametrize("paths", [1, 129, 300])
@pytest.mark.parametrize("scheme", ["full", "picard"])
def test_swaptions_with_two_paths_a_thread_and_a_ragged_tile(lll, paths, scheme):
    wl = _flat(34, 5, 64, 0.1)
    x, W = quadrature.rule_for(wl)
    _check(lll, wl, x, W, scheme, paths, (64, 0, 0, 2, 1), product="swaption")


@pytest.mark.parametrize("scheme,mapping,launch", [("full", "path", None), ("picard", "path", None), ("full", "path", ONE_LANE),
                                                   ("picard", "step", ONE_LANE)])
def test_volatilities_of_both_signs(lll, scheme, mapping, launch):
    wl = _flat(20, 4, 64, 0.15)
    sign = np.where(np.arange(wl.n) % 3 == 1, -1.0, 1.0)
    wl = dataclasses.replace(wl, lam=wl.lam * sign)
    x, W = quadrature.rule_for(wl)
    lam = wl.lam[0]
    assert len(lll.lll_sweep_rule(x, W, lam[lam < 0].sum(), lam[lam > 0].sum())[0]) > 0
    _check(lll, wl, x, W, scheme, 500, launch, mapping)


@pytest.mark.parametrize("paths", [116736, 116737, 150001])
@pytest.mark.parametrize("launch", [None, (64, 0, 0, 1, 1)])
def test_frozen_drift_on_both_sides_of_its_two_kernels(lll, paths, launch):
    """The last 64 paths of a launch against the oracle, and its sums against those of the
    same paths in three smaller launches."""
    wl = _flat(6, 3, 32, 0.15)
    x, W = quadrature.rule_for(wl)
    sim = lll.LevyLibor(wl, x, W)
    try:
        if launch:
            sim.set_launch(*launch)
        sim.simulate("frozen", paths=paths)
        s1, s2, _ = sim.sums()
        p1, p2 = np.zeros_like(s1), np.zeros_like(s2)
        cuts = [0, paths // 3, 2 * (paths // 3), paths - 64, paths]
        for a, b in zip(cuts, cuts[1:]):
            sim.simulate("frozen", paths=b - a, first_path=a, snapshots=64)
            z = sim.paths(0, 64).astype(np.float64)
            u1, u2, _ = sim.sums()
            p1, p2 = p1 + u1, p2 + u2
    finally:
        sim.close()
    assert np.allclose(s1, p1, rtol=1e-12, atol=0) and np.allclose(s2, p2, rtol=1e-12, atol=0)
    ref = ora.simulate(ora.OracleModel(wl, x, W), ora.FROZEN, path0=paths - 64, npaths=64, want_snap=True)
    mask = ~np.isnan(ref["snap"])
    assert np.abs(np.expm1(z[mask] - ref["snap"][mask])).max() <= 1e-5
