"""The FP64 helpers that stand in for CUDA's functions (csrc/pdq_device.cuh, csrc/pdq_lf_math.cuh), each swept over its
argument range beside the function it replaces.  Bars in units of 2^-53 of the value, from the roundings of both sides
and the truncation that the helper states."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_04979_gb300 import build as b
    out = str(tmp_path_factory.mktemp("math64") / "check.so")
    subprocess.run([b.nvcc()] + b.ARCH + ["-O3", "-std=c++17", "-I", b.CSRC, "-I", os.path.join(b.ROOT, "include"),
                                          "-Xcompiler", "-fPIC", "-shared", "-cudart", "shared", "-o", out,
                                          os.path.join(HERE, "math64_check.cu")], check=True, capture_output=True)
    return ctypes.CDLL(out)


def _both(lib, x, a):
    """out[k, 0] ours and out[k, 1] CUDA's, k as in math64_check.cu."""
    n = len(x)
    xs, av = torch.tensor(x, device="cuda"), torch.tensor(a, device="cuda")
    out = torch.empty((5, 2, n), dtype=torch.float64, device="cuda")
    p = ctypes.c_void_p
    assert lib.check_math(p(xs.data_ptr()), p(av.data_ptr()), n, p(out.data_ptr())) == 0
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _units(o, k):
    return float(np.max(np.abs(o[k, 0] / o[k, 1] - 1))) * 2.0 ** 53


def test_estimates(lib):
    # arguments over 2^-80 .. 2^80, the mantissas at random and at both ends of the 20 bits that the estimates see
    rng = np.random.default_rng(1)
    m = np.r_[1 + rng.random(200000), 1 + np.arange(4096) / 4096, np.nextafter(1 + np.arange(1, 4097) / 4096, 0)]
    x = m * 2.0 ** rng.integers(-80, 81, m.size)
    o = _both(lib, x, np.ones_like(x))
    assert _units(o, 0) <= 2.0 ** (53 - 19) and _units(o, 1) <= 2.0 ** (53 - 19)


def test_root_of_the_momentum_equation(lib):
    # a = dy/tau and c over the ranges that grids and classes span, far beyond either side of a^2 = 2c.  Ours: 1 from
    # u/2 + a, 1 of the result, 2^-55 truncation; the closed form: half of a^2 + 2c's, 1 each of root, sum and quotient
    rng = np.random.default_rng(2)
    a, c = 10.0 ** rng.uniform(-8, 4, 400000), 10.0 ** rng.uniform(-20, 6, 400000)
    assert _units(_both(lib, c, a), 2) <= 6


def test_exponential_quotient(lib):
    # -x from 1e-12 over both polynomials' ends and the step to the library's exponential to -40.  Ours: below 1/2 two
    # roundings and 2^-57; beyond, exp's ulp over e^-x - 1 (2.5 units) and the quotient; CUDA's expm1 1 ulp, a quotient
    rng = np.random.default_rng(3)
    ends = np.array([0.015625, 0.5])
    x = np.r_[10.0 ** rng.uniform(-12, np.log10(40), 400000), rng.uniform(0.01, 0.6, 100000), ends,
              np.nextafter(ends, 0), np.nextafter(ends, 1)]
    o = _both(lib, x, np.ones_like(x))
    assert _units(o, 3) <= 7 and _units(o, 4) <= 4
