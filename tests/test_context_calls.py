"""What the calls of a context ask of the CUDA runtime: the host code of the C ABI
on a fake runtime and fake launchers (tests/host_helpers), on the CPU."""
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
    exe = str(tmp_path_factory.mktemp("context") / "context_calls")
    # launchers that no check reaches stay undefined
    subprocess.check_call([cxx, "-std=c++17", "-O1", "-D_GLIBCXX_ASSERTIONS", "-I", cuda + "/include", "-I",
                           os.path.join(ROOT, "include"), "-Wl,--unresolved-symbols=ignore-all", "-Wl,-z,lazy", "-no-pie", "-o",
                           exe, os.path.join(HERE, "host_helpers", "context_calls.cpp")])
    return exe


@pytest.mark.parametrize("what", ["compensators", "selections", "fewer_paths", "limits", "batch_limits"])
def test_context_calls(helper, what):
    r = subprocess.run([helper, what], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stderr)
