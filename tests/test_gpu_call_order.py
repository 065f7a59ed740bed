"""What a context was asked before must not change what it answers: selecting a
mapping and setting it back, and the same selections inside a stream capture."""
import numpy as np
import pytest

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


SELECT = {"tenor": lambda sim: sim.set_mapping("tenor", 8), "lanes": lambda sim: sim.set_launch(0, 0, 0, 0, 2)}
BACK = {"tenor": lambda sim: sim.set_mapping("path"), "lanes": lambda sim: sim.set_launch()}


@pytest.mark.parametrize("maker,hidden,layers,head", [(workloads.large_single, 128, 3, 0), (workloads.large_single, 128, 3, 1),
                                                      (workloads.long_dated, 256, 4, 1)])
@pytest.mark.parametrize("how", ["tenor", "lanes"])
def test_learned_drift_prices_do_not_depend_on_earlier_selections(env, maker, hidden, layers, head, how):
    _, lll = env
    sim = lll.LevyLibor(maker(paths=2000))
    try:
        lll.lll_mlp_init_head(sim.ctx, hidden, layers, head, 3)
        p, sc = lll.lll_mlp_params(sim.ctx, 0, count=lll.lll_mlp_layout(sim.ctx, layers)[0])
        sc[4] = 1e-3  # the target unit of a trained network
        lll.lll_mlp_params(sim.ctx, 1, p, scales=sc)
        sim.simulate("mlp", snapshots=2000)
        z, sums = sim.paths(0, 2000), sim.sums()
        SELECT[how](sim)
        sim.simulate("picard")
        BACK[how](sim)
        sim.simulate("mlp", snapshots=2000)
        z2, sums2 = sim.paths(0, 2000), sim.sums()
    finally:
        sim.close()
    assert np.array_equal(z, z2, equal_nan=True)
    assert np.array_equal(sums[0], sums2[0]) and np.array_equal(sums[1], sums2[1])


@pytest.mark.parametrize("how", ["tenor", "lanes"])
def test_selection_inside_a_capture(env, how):
    """The selection and the simulation captured into one graph: the graph gives the
    sums of the same calls outside, and the context is sound afterwards."""
    torch, lll = env
    wl = workloads.large_single(paths=3000)
    stream = torch.cuda.Stream()
    ref, sim = lll.LevyLibor(wl), lll.LevyLibor(wl, stream=stream.cuda_stream)
    out = torch.zeros((wl.n, wl.strikes.shape[1], 2), dtype=torch.float64, device="cuda")
    noalloc = lambda s, seed: lll.lll_simulate_noalloc(s.ctx, lll.LLL_PICARD, 0, wl.paths, seed, out.data_ptr())  # noqa: E731
    try:
        SELECT[how](ref)
        ref.simulate("picard", seed=5)
        want = ref.sums()
        noalloc(sim, 1)  # finds the scratch array
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            SELECT[how](sim)
            noalloc(sim, 5)
        for _ in range(2):
            out.fill_(float("nan"))
            graph.replay()
            torch.cuda.synchronize()
            assert np.allclose(out[..., 0].cpu().numpy(), want[0], rtol=1e-12, atol=0)
            assert np.allclose(out[..., 1].cpu().numpy(), want[1], rtol=1e-12, atol=0)
        sim.simulate("picard", seed=5)
        got = sim.sums()
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    finally:
        ref.close()
        sim.close()
