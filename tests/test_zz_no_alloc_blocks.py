"""lll_simulate_noalloc where the scratch of lll_simulate's launch is larger than the
static array, although that of the rule as given is not: fewer blocks run, or the
time-blocked kernel in place of the pipeline, and the sums agree to the grouping of
their FP64 partials (1e-12, as in test_zz_no_alloc.py)."""
import dataclasses

import numpy as np
import pytest

from paper_1006_3340_gb300 import workloads

pytestmark = pytest.mark.gpu

MANY = np.linspace(0.02, 0.08, 50)


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1006_3340_gb300 import lll

    lll.load()
    return torch, lll


@pytest.mark.parametrize("maker,scheme,paths,strikes,launch", [
    (workloads.large_single, "picard", 1 << 18, None, None),                  # state of all blocks, two paths a thread
    (workloads.long_dated, "full", 20001, MANY, (128, 1, 0, 1, 1)),           # state and payoff sums
    (workloads.long_dated, "full", 60001, MANY, None),                        # payoff sums alone
    (workloads.long_dated, "full", 12000, MANY, None)])                       # the pipeline's payoff sums
@pytest.mark.parametrize("product", ["caplet", "swaption"])
def test_more_scratch_than_the_static_array(env, maker, scheme, paths, strikes, launch, product):
    torch, lll = env
    wl = maker(paths=paths)
    if strikes is not None:
        wl = dataclasses.replace(wl, strikes=np.tile(strikes, (wl.n, 1)))
    sim = lll.LevyLibor(wl)
    try:
        sim.set_product(product)
        if launch is not None:
            sim.set_launch(*launch)
        sim.simulate(scheme)
        s1, s2, _ = sim.sums()
        out = torch.full((wl.n, wl.strikes.shape[1], 2), float("nan"), dtype=torch.float64, device="cuda")
        lll.lll_simulate_noalloc(sim.ctx, lll.SCHEMES[scheme], 0, wl.paths, wl.seed, out.data_ptr())
        torch.cuda.synchronize()
        got = out.cpu().numpy()
    finally:
        sim.close()
    for g, s in ((got[..., 0], s1), (got[..., 1], s2)):
        assert np.allclose(g, s, rtol=1e-12, atol=0)
