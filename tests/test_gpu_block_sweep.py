"""The time-blocked sweep (lll_paths_block.cu) where it can go wrong, path by
path against the FP64 oracle on the rule as given: steps per period that are
not a multiple of the block length, one rate, chunks shorter than the live
rates, ragged path tiles, every padded node count, one and two paths per
thread, and a batch whose instances sweep rules of different lengths, or, with
a signed rule among them, the rules as given.  Bars as in test_gpu_parity.py
(FP32 path state: 1e-5 on rates, 1e-7 on prices)."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as ora
from oracle import quadrature
from paper_1006_3340_gb300 import workloads

pytestmark = pytest.mark.gpu
SCHEMES = {"full": ora.FULL, "picard": ora.PICARD}


@pytest.fixture(scope="module")
def lll():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1006_3340_gb300 import lll as mod

    mod.load()
    return mod


def _check(lll, wl, x, W, scheme, paths, launch):
    sim = lll.LevyLibor(wl, x, W)
    try:
        sim.set_launch(*launch)
        sim.simulate(scheme, paths=paths, snapshots=paths)
        z = sim.paths(0, paths).astype(np.float64)
        p, _ = sim.prices()
    finally:
        sim.close()
    ref = ora.simulate(ora.OracleModel(wl, x, W), SCHEMES[scheme], npaths=paths, want_snap=True)
    mask = ~np.isnan(ref["snap"])
    assert np.array_equal(mask, ~np.isnan(z))
    assert np.abs(np.expm1(z[mask] - ref["snap"][mask])).max() <= 1e-5
    assert np.abs(p - ref["price"]).max() <= 1e-7


# (N, s, volatility level, padded nodes expected): steeper volatilities need longer rules
SHAPES = [(2, 1, 0.12, 4), (3, 7, 0.12, 4), (5, 9, 0.12, 4), (41, 3, 0.05, 8), (34, 5, 0.15, 12), (40, 2, 0.24, 16),
          (60, 3, 0.27, 20), (70, 2, 0.28, 24)]


@pytest.mark.parametrize("N,s,level,padded", SHAPES)
@pytest.mark.parametrize("scheme", ["full", "picard"])
@pytest.mark.parametrize("launch", [(32, 0, 1, 1, 1), (64, 1, 0, 2, 1), (128, 0, 5, 0, 1)])
def test_shapes_and_lengths(lll, N, s, level, padded, scheme, launch):
    wl = workloads.tiny(N=N, s=s, Q=64)
    wl = dataclasses.replace(wl, lam=np.full_like(wl.lam, level), L0=np.full(N, 0.03))
    x, W = quadrature.rule_for(wl)
    assert lll.lll_sweep_rule(x, W, 0.0, level * wl.n)[2] == padded
    _check(lll, wl, x, W, scheme, 75, launch)


@pytest.mark.parametrize("scheme", ["full", "picard"])
def test_longest_rule(lll, scheme):
    wl = workloads.paper_example()  # heavy tails, nodes up to |x| = 30
    x, W = quadrature.rule_for(wl)
    assert lll.lll_sweep_rule(x, W, 0.0, wl.lam.sum(1).max())[2] == 32
    _check(lll, wl, x, W, scheme, 300, (64, 0, 0, 1, 1))


@pytest.mark.parametrize("paths", [1, 33, 5000])
def test_path_counts_default_launch(lll, paths):
    wl = workloads.tiny(N=6, s=10, Q=32)
    x, W = quadrature.rule_for(wl)
    _check(lll, wl, x, W, "full", paths, (0, 0, 0, 0, 0))


@pytest.mark.parametrize("levels", [(0.05, 0.05, 0.05), (0.05, 0.15, 0.3), (0.05, 0.15, None)])
@pytest.mark.parametrize("scheme", ["full", "picard"])
@pytest.mark.parametrize("ppt", [1, 2])
def test_batch_of_rule_lengths(lll, levels, scheme, ppt):
    inst = []
    for q, level in enumerate(levels):
        wl = workloads.tiny(N=8 + 20 * q, s=3, Q=64, paths=100 + 61 * q)
        wl = dataclasses.replace(wl, lam=np.full_like(wl.lam, level or 0.15), L0=np.full(wl.N, 0.03))
        x, W = quadrature.rule_for(wl)
        if level is None:  # a signed rule: split one node's weight into 1.5 and -0.5 of it
            j = np.argmin(np.abs(x))
            x, W = np.append(x[1:], x[j]), np.append(W[1:], -0.5 * W[j])
            W[j - 1] *= 1.5
        inst.append((wl, x, W))
    b, keep = lll.lll_batch_init(inst)
    try:
        lll.lll_batch_set_launch(b, 64, 0, 0, ppt)
        lll.lll_batch_simulate(b, lll.SCHEMES[scheme], 11)
        got = [lll.lll_batch_prices(b, q, wl.n, wl.strikes.shape[1])[0] for q, (wl, _, _) in enumerate(inst)]
    finally:
        lll.lll_batch_destroy(b)
    for q, (wl, x, W) in enumerate(inst):
        ref = ora.simulate(ora.OracleModel(wl, x, W), SCHEMES[scheme], seed=11, inst=q)
        assert np.abs(got[q] - ref["price"]).max() <= 1e-7, q


# The pipeline for few paths (lll_paths_pipe.cu): the same arithmetic, so its
# recorded log-rates equal the block kernel's bit for bit, and its sums differ
# only by their double-float order.
@pytest.mark.parametrize("N,s,level", [(2, 1, 0.12), (4, 8, 0.12), (9, 5, 0.1), (10, 10, 0.12), (18, 3, 0.12),
                                       (41, 8, 0.05), (34, 5, 0.15), (40, 3, 0.24), (120, 4, 0.02), (60, 4, 0.27),
                                       (70, 2, 0.28)])
@pytest.mark.parametrize("scheme", ["full", "picard"])
@pytest.mark.parametrize("paths", [1, 70, 5000])
def test_pipeline_equals_block_kernel(lll, N, s, level, scheme, paths):
    wl = workloads.tiny(N=N, s=s, Q=64)
    wl = dataclasses.replace(wl, lam=np.full_like(wl.lam, level), L0=np.full(N, 0.03))
    x, W = quadrature.rule_for(wl)
    got = []
    for launch in ((0, 0, 0, 0, 0), (64, 0, 0, 1, 1)):
        sim = lll.LevyLibor(wl, x, W)
        try:
            sim.set_launch(*launch)
            sim.simulate(scheme, paths=paths, snapshots=min(paths, 200), snapshot_stride=7 if paths > 1400 else 1)
            got.append((sim.paths(0, min(paths, 200)), *sim.sums()))
        finally:
            sim.close()
    assert np.array_equal(got[0][0], got[1][0], equal_nan=True)
    for u, v in ((got[0][1], got[1][1]), (got[0][2], got[1][2])):
        assert np.all(np.abs(u - v) <= 1e-12 * np.abs(v))
