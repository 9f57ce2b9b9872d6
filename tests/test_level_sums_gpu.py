"""The FP32 form's weighted sums over delayed levels (level_sums.cuh) against extended precision."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2506_03027_gb300", "csrc")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("sums") / "libsums.so")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "--fmad=false", "-shared", "-Xcompiler",
                    "-fPIC", "-I", CSRC, os.path.join(HERE, "cuda", "level_sums_check.cu"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    lib.level_sums.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
    return lib


def extrapolation(k):
    """Lagrange weights of the levels -k, .., -(k + 4) at one step ahead of level 0."""
    t = -(k + np.arange(5, dtype=np.longdouble))
    return np.array([np.prod([(1 - t[j]) / (t[l] - t[j]) for j in range(5) if j != l]) for l in range(5)]).astype(np.float64)


# the largest delay, where sum |W| is largest; levels of one sign and size, and levels that change sign
@pytest.mark.parametrize("k", [0, 4])
@pytest.mark.parametrize("base,change", [(1.0, 1e-3), (2e-3, 5e-3), (0.0, 1.0)])
def test_sums_over_levels(lib, k, base, change):
    import torch
    rng = np.random.default_rng(17)
    n = 1 << 14
    t = -(k + np.arange(5.0))
    b = base * rng.uniform(0.5, 1.0, (n, 1, 5)) * rng.choice([-1.0, 1.0], (n, 1, 5))
    r = b + change * (rng.uniform(-1, 1, (n, 1, 5)) * t[None, :, None] + 0.01 * rng.uniform(-1, 1, (n, 1, 5)) * t[None, :, None] ** 2)
    W = extrapolation(k)
    c = np.array([W.sum() - 1.0, *W[1:]])
    hi = c.astype(np.float32)
    pairs = np.stack([hi, (c - hi).astype(np.float32)], 1)
    rt, ct = torch.tensor(r, device="cuda"), torch.tensor(pairs, device="cuda")
    out = torch.empty((n, 5), dtype=torch.float32, device="cuda")
    assert lib.level_sums(rt.data_ptr(), ct.data_ptr(), out.data_ptr(), n) == 0
    R = r.astype(np.longdouble)
    ref = (c.astype(np.longdouble)[1:, None] * (R[:, 1:] - R[:, :1])).sum(axis=1) + np.longdouble(c[0]) * R[:, 0]
    # the sum's own rounding to FP32, and a few roundings to 2^-48 of the levels and weights
    tol = 2.0 ** -24 * np.abs(ref) + 8 * 2.0 ** -48 * np.abs(W).sum() * np.abs(R).max(axis=1)
    err = np.abs(out.cpu().numpy().astype(np.longdouble) - ref)
    assert np.all(err <= tol), float((err / tol).max())
