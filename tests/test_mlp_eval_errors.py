"""lll_mlp_eval's host code on a fake CUDA runtime (tests/host_helpers), on the
CPU: what a failing call leaves behind.  An evaluation whose n-th call fails
reports it and returns with no work in flight on either of its streams (its
copies read and write the caller's arrays); one that could not create an event
leaves a network that the next evaluation can use."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def helper(tmp_path_factory):
    cxx = shutil.which("g++")
    cuda = next((d for d in (os.environ.get("CUDA_HOME"), "/usr/local/cuda") if d and os.path.exists(d + "/include/cuda_runtime.h")),
                None)
    if cxx is None or cuda is None:
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("mlp_eval") / "mlp_eval_errors")
    # launchers that an evaluation does not reach stay undefined
    subprocess.check_call([cxx, "-std=c++17", "-O1", "-D_GLIBCXX_ASSERTIONS", "-I", cuda + "/include", "-I",
                           os.path.join(ROOT, "include"), "-Wl,--unresolved-symbols=ignore-all", "-Wl,-z,lazy", "-no-pie", "-o",
                           exe, os.path.join(HERE, "host_helpers", "mlp_eval_errors.cpp")])
    return exe


@pytest.mark.parametrize("n", range(1, 6))
def test_failed_event_leaves_a_usable_network(helper, n):
    r = subprocess.run([helper, "events", str(n)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stderr)


def test_failed_call_returns_with_nothing_in_flight(helper):
    r = subprocess.run([helper, "calls"], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stderr)
