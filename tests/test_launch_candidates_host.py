"""Launch candidates that name a mapping must run it: with the default launch shape
the step mapping may run the path mapping's kernels."""
import bench
from paper_1006_3340_gb300 import autotune


def _step(cands):
    return [c for c in cands if len(c) > 5 and c[5] < 0]


def test_step_parallel_candidates_have_a_launch_shape_of_their_own():
    for cands in (list(autotune.DEFAULT_CANDIDATES), [c for _, c in bench.MAPPING_SHAPES]):
        assert _step(cands)
        for c in _step(cands):
            assert c[0] > 0 and c[3] == 1 and c[4] == 1, c
