"""The step mapping of a default launch takes the faster kernels: the step kernels
where few paths leave the path mapping's waiting, the path mapping's where paths
fill the GPU.  Device times of the two differ by 1.8 to 15 times on these shapes; the
bars ask for a third of the saving."""
import dataclasses

import numpy as np
import pytest

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


def _flat(N, s, level):
    wl = workloads.tiny(N=N, s=s, Q=64)
    return dataclasses.replace(wl, lam=np.full_like(wl.lam, level), L0=np.full(N, 0.03))


def _ms(sim, paths, launch, mapping):
    sim.set_launch(*launch)
    sim.set_mapping(mapping)
    t = []
    for _ in range(7):
        sim.simulate("picard", paths=paths)
        t.append(sim.kernel_ms()[1])
    return float(np.median(t[2:]))


DEFAULT, ONE_LANE = (0, 0, 0, 0, 0), (128, 0, 0, 1, 1)


@pytest.mark.parametrize("wl,paths", [(_flat(120, 8, 0.02), 100), (_flat(120, 8, 0.02), 2000), (_flat(20, 100, 0.1), 300),
                                      (_flat(2, 500, 0.1), 500), (_flat(300, 1, 0.02), 1000), (workloads.long_dated(), 300)])
def test_few_paths_take_the_step_kernels(lll, wl, paths):
    sim = lll.LevyLibor(wl)
    try:
        path, step = _ms(sim, paths, DEFAULT, "path"), _ms(sim, paths, DEFAULT, "step")
    finally:
        sim.close()
    assert step < path - (1 - 1 / 1.8) / 3 * path, (path, step)


@pytest.mark.parametrize("wl,paths", [(workloads.large_single(), 4096), (workloads.large_single(), 64000),
                                      (_flat(120, 8, 0.02), 64000)])
def test_many_paths_take_the_path_kernels(lll, wl, paths):
    sim = lll.LevyLibor(wl)
    try:
        kernels, default = _ms(sim, paths, ONE_LANE, "step"), _ms(sim, paths, DEFAULT, "step")
    finally:
        sim.close()
    assert default < kernels - (1 - 1 / 1.8) / 3 * kernels, (kernels, default)
