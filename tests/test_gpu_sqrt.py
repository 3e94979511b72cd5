"""The integer-pipe square root of the Newton kernels must equal CUDA's
correctly rounded __dsqrt_rn bit for bit: every leading significand (one
binary32 seed each) for both parities of the exponent, random bit patterns,
squares and their neighbours (the results closest to a rounding boundary), and
the values that take the fallback."""
import ctypes
import os
import subprocess
import tempfile

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def helper():
    out = os.path.join(tempfile.mkdtemp(), "sqrt_check.so")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "-I" + os.path.join(ROOT, "include"), "-Xcompiler", "-fPIC", "-shared",
                    os.path.join(ROOT, "tests", "gpu_helpers", "sqrt_check.cu"), "-o", out],
                   check=True, capture_output=True)
    lib = ctypes.CDLL(out)
    lib.sqrt_check.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int64]
    return lib


def check(helper, x):
    d = torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()
    o, r = torch.empty_like(d), torch.empty_like(d)
    assert helper.sqrt_check(d.data_ptr(), o.data_ptr(), r.data_ptr(), d.numel()) == 0
    o, r = o.cpu().numpy(), r.cpu().numpy()
    bad = (o.view(np.uint64) != r.view(np.uint64)) & ~(np.isnan(o) & np.isnan(r))
    assert not bad.any(), f"{bad.sum()} mismatches, e.g. x={x[bad][:3]!r}"


@pytest.mark.parametrize("exponent", [1022, 1023])
@pytest.mark.parametrize("low", ["zero", "ones", "random"])
def test_every_seed(helper, exponent, low):
    g = np.random.Generator(np.random.Philox(41))
    top = np.arange(1 << 23, dtype=np.uint64) << np.uint64(29)
    tail = {"zero": np.uint64(0), "ones": np.uint64((1 << 29) - 1),
            "random": g.integers(0, 1 << 29, size=1 << 23, dtype=np.uint64)}[low]
    check(helper, (np.uint64(exponent << 52) | top | tail).view(np.float64))


def test_random_and_boundaries(helper):
    g = np.random.Generator(np.random.Philox(42))
    check(helper, g.integers(0, 2 ** 63, size=1 << 24, dtype=np.uint64).view(np.float64))
    # (s + half a unit)^2 and s^2, rounded, with their neighbours
    s = 1.0 + g.random(1 << 20)
    for v in (s * s, s * s + s * 2.0 ** -52):
        for k in (-2, -1, 0, 1, 2):
            check(helper, (v.view(np.int64) + k).view(np.float64))
    check(helper, np.array([0.0, -0.0, 1.0, 4.0, 2.0, np.inf, -np.inf, np.nan, -1.0, 5e-324, 2.2250738585072014e-308,
                            2.2250738585072009e-308, 1.7976931348623157e308, 3.9999999999999996, 0.9999999999999999]))
