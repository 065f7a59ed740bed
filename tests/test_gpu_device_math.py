"""The FP32 division and square root of the sampler, and the root of the inverse
Gaussian draw, against FP64 on the device.

Bounds: both operations claim one ulp (one correction step from approximations of
1 and 2 ulp leaves half an ulp of rounding and about 2^-44 of the value), over the
whole range of operands, on both sides of the points where they hand over to the
full-range operations.  The root must be the one that FP64 takes, always."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1006_3340_gb300 import workloads

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available to build the helper")
    so = str(tmp_path_factory.mktemp("device_math") / "libdevice_math.so")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                           "-fPIC", "-o", so, os.path.join(HERE, "gpu_helpers", "device_math.cu")])
    lib = ctypes.CDLL(so)
    V, D, I, U = ctypes.c_void_p, ctypes.c_double, ctypes.c_int, ctypes.c_uint
    lib.device_math.argtypes = [I, V, V, I, V]
    lib.device_roots.argtypes = [D, D, D, D, U, U, I, D, V, V, V]
    return lib


def _errors(dev, what, a, b):
    a, b = (np.ascontiguousarray(v, dtype=np.float32) for v in (a, b))
    err = np.zeros(len(a))
    assert dev.device_math(what, a.ctypes.data, b.ctypes.data, len(a), err.ctypes.data) == 0
    return err


def _spread(rng, lo, hi, count):
    """Positive numbers, evenly over the logarithm, the ends and their neighbours among them."""
    v = np.exp(rng.uniform(np.log(lo), np.log(hi), count)).astype(np.float32)
    ends = np.float32([lo, hi])
    v[:6] = np.concatenate([ends, np.nextafter(ends, np.float32(0)), np.nextafter(ends, np.float32(np.inf))])
    return v


# numerators down to the smallest normal number and into the denormal ones
@pytest.mark.parametrize("a", [(1e-6, 1e2), (1e-30, 1e-6), (1e-38, 1e-30), (1e-44, 1e-38), (1e2, 1e18), (1e18, 3e38)])
@pytest.mark.parametrize("b", [(1e-6, 1e2), (9e-19, 1.1e-18), (9e17, 1.1e18), (1e-18, 1e18), (1e-37, 1e37)])
def test_quotient_is_within_one_ulp(dev, a, b):
    rng = np.random.default_rng(3)
    x, y = _spread(rng, *a, 1 << 18), _spread(rng, *b, 1 << 18)
    rng.shuffle(y)
    with np.errstate(all="ignore"):
        fits = x.astype(np.float64) / y.astype(np.float64) < 3.4e38
    assert fits.any() or a[0] > 1 or b[1] < 1
    err = _errors(dev, 0, x[fits], y[fits]) if fits.any() else np.zeros(1)
    assert err.max() <= 1.0


@pytest.mark.parametrize("x", [(1e-6, 1e2), (9e-31, 1.1e-30), (9e29, 1.1e30), (1e-30, 1e30), (1e-44, 3e38)])
def test_square_root_is_within_one_ulp(dev, x):
    rng = np.random.default_rng(4)
    v = _spread(rng, *x, 1 << 18)
    assert _errors(dev, 1, v, v).max() <= 1.0


@pytest.mark.parametrize("maker", [workloads.small_plain, workloads.large_single, workloads.long_dated, workloads.paper_example])
def test_root_of_the_inverse_gaussian_draw_is_the_one_of_fp64(dev, maker):
    wl = maker()
    gam = np.sqrt(wl.alpha ** 2 - wl.beta ** 2)
    h = wl.delta / wl.s
    wrong, near, differ, total = ctypes.c_ulonglong(), ctypes.c_ulonglong(), ctypes.c_ulonglong(), 0
    for k in range(4):
        rc = dev.device_roots(wl.dbar * h / gam, (wl.dbar * h) ** 2, wl.beta, -wl.dbar * wl.beta / gam * h, 17, k, 1 << 23, 4e-5,
                              ctypes.addressof(wrong), ctypes.addressof(near), ctypes.addressof(differ))
        assert rc == 0
        assert wrong.value == 0 and differ.value == 0
        total += near.value
    assert total > 100  # the band in which FP32 and FP64 could differ has been drawn
