"""newton_tile (csrc/pdq_newton.cuh) at every width and cut that its launches can take, compiled here with the cut given,
against the direct sum in float64."""
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
    out = str(tmp_path_factory.mktemp("tile") / "check.so")
    subprocess.run([b.nvcc()] + b.ARCH + ["-O3", "-std=c++17", "-I", b.CSRC, "-I", os.path.join(b.ROOT, "include"),
                                          "-Xcompiler", "-fPIC", "-shared", "-cudart", "shared", "-o", out,
                                          os.path.join(HERE, "newton_tile_check.cu")], check=True, capture_output=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("NT", [64, 128])
@pytest.mark.parametrize("U", [4, 8, 12])
@pytest.mark.parametrize("sizes", ["1", "T-1", "T", "T+1", "2*T+1"])
def test_sums_of_given_cuts(lib, NT, U, sizes):
    # one sample of one particle, one tile -1, exactly, +1 and two tiles +1 (the edge between a tile's own block and the
    # later particles), whole and in 2, 3 and more parts than there are j-tiles; z-sorted like a binned sample.  One
    # charged particle at a time, at the edges of groups, tiles and parts: every other particle's sum is that one term,
    # once, and nothing else.  Bar: r^2 to 3 2^-24, its power -3/2 to 9, the products to 4: 16 2^-24 of the term; the
    # separations to 2^-24 of coordinates up to 720: another 4 x 720 2^-24 / r of it
    T = NT * U
    n = eval(sizes, {"T": T})
    rng = np.random.default_rng(n)
    r, th = 178.0 * np.sqrt(rng.random(n)), 2 * np.pi * rng.random(n)
    pos = torch.tensor(np.stack([r * np.cos(th), r * np.sin(th), np.sort(720.0 * rng.random(n)), np.zeros(n)], 1),
                       dtype=torch.float32, device="cuda")
    ptr = ctypes.c_void_p
    for j in sorted({k for k in (0, 31, 32, 32 * U, T // 2, T - 1, T, T + NT - 1, T + NT, n - 1) if k < n}):
        q = 0.5 + 0.5 * rng.random()
        pos[:, 3] = 0.0
        pos[j, 3] = q
        p = pos.double()
        d = p[:, :3] - p[j, :3]
        d[:, 2] -= 720.0 * torch.round(d[:, 2] / 720.0)
        r2 = torch.clamp((d * d).sum(1), min=0.09)
        want = p[j, 3] * d / (r2 * torch.sqrt(r2))[:, None]
        bar = (16 + 4 * 720.0 / torch.sqrt(r2)) * 2.0 ** -24 * want.norm(dim=1)
        for parts in (1, 2, 3, n // NT + 4):
            acc = torch.zeros((n, 4), dtype=torch.float32, device="cuda")
            assert lib.check_tile(ptr(pos.data_ptr()), ptr(acc.data_ptr()), n, NT, U, parts, ctypes.c_float(720.0),
                                  ctypes.c_float(0.09)) == 0
            torch.cuda.synchronize()
            assert bool(torch.all((acc[:, :3].double() - want).norm(dim=1) <= bar)), (j, parts)
            assert bool(torch.all(acc[j] == 0)), (j, parts)
