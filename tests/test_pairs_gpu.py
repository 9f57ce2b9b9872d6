"""The arithmetic on pairs of floats (pairs.cuh) against extended precision, element by element."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2506_03027_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("pairs") / "libpairs.so")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "-I", CSRC, os.path.join(HERE, "cuda", "pairs_check.cu"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    lib.pairs_check.argtypes = [ctypes.c_void_p] * 5 + [ctypes.c_int]
    lib.pairs_pow.argtypes = [ctypes.c_void_p, ctypes.c_double, ctypes.c_void_p, ctypes.c_int]
    return lib


# values near 1, over many magnitudes, and sums that cancel almost entirely
@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["unit", "wide", "cancel"])
def test_pair_operations(lib, kind):
    import torch
    rng = np.random.default_rng(11)
    n = 1 << 18
    a, b, c = (rng.choice([-1.0, 1.0], n) * rng.uniform(0.5, 2.0, n) for _ in range(3))
    if kind == "wide":
        a, b, c = (x * 10.0 ** rng.uniform(-9, 9, n) for x in (a, b, c))
    if kind == "cancel":
        b = a * (1.0 + 10.0 ** rng.uniform(-14, -3, n))
        c = -a * b * (1.0 + 10.0 ** rng.uniform(-14, -3, n))
    t = [torch.tensor(x, device="cuda") for x in (a, b, c)]
    out = torch.empty((7, n, 2), dtype=torch.float32, device="cuda")
    dbl = torch.empty(n, dtype=torch.float64, device="cuda")
    assert lib.pairs_check(*(x.data_ptr() for x in t), out.data_ptr(), dbl.data_ptr(), n) == 0
    got = out.cpu().numpy().astype(np.longdouble).sum(axis=-1)
    a, b, c = (x.astype(np.longdouble) for x in (a, b, c))
    u = np.longdouble(2.0) ** -48
    # h to 24 bits and l to 24 bits of what is left; the other operations on split operands (each off by
    # u/2) with a handful of roundings of low words, u/2 of the operands' magnitudes each
    exact = [(a, u / 2 * abs(a)), (a + b, 3 * u * (abs(a) + abs(b))), (a - b, 3 * u * (abs(a) + abs(b))),
             (a * b, 4 * u * abs(a * b)), (a * b + c, 6 * u * (abs(a * b) + abs(c))), (1 / a, 4 * u / abs(a)),
             (a * b + c, 6 * u * (abs(a * b) + abs(c)))]
    for k, (ref, tol) in enumerate(exact):
        assert np.all(abs(got[k] - ref) <= tol), (k, float(np.max(abs(got[k] - ref) / tol)))
    assert np.all(dbl.cpu().numpy().astype(np.longdouble) == got[0])  # 48 bits and a sign: exact in FP64


@pytest.mark.gpu
def test_split_outside_the_fp32_range(lib):
    """Nonfinite values and values beyond FP32 give NaN, values below it zero."""
    import torch
    x = np.array([np.nan, np.inf, -np.inf, 1e39, -1e200, 1e-39, -1e-300, 0.0, -0.0, 1e38, 2.0 ** -126])
    t = torch.tensor(x, device="cuda")
    one = torch.ones_like(t)
    out = torch.empty((7, len(x), 2), dtype=torch.float32, device="cuda")
    dbl = torch.empty(len(x), dtype=torch.float64, device="cuda")
    assert lib.pairs_check(t.data_ptr(), one.data_ptr(), one.data_ptr(), out.data_ptr(), dbl.data_ptr(), len(x)) == 0
    d = dbl.cpu().numpy()
    assert np.all(np.isnan(d[:5])) and np.all(d[5:9] == 0.0)
    assert abs(d[9] - 1e38) <= 2.0 ** -49 * 1e38 and d[10] == 2.0 ** -126


@pytest.mark.gpu
@pytest.mark.parametrize("a", [0.76, -0.76, 1.5, 0.001])
def test_power(lib, a):
    """x^a near 1 (every table entry, both sides of 1), over the FP32 range, and where it falls back."""
    import torch
    rng = np.random.default_rng(13)
    x = np.concatenate([1.0 + rng.uniform(-0.05, 0.05, 1 << 16), rng.uniform(0.2, 4.0, 1 << 16), 300.0 * rng.uniform(0.5, 2.0, 1 << 16),
                        10.0 ** rng.uniform(-30, 30, 1 << 16), 1.0 + np.array([0.0, 2.0 ** -30, -2.0 ** -30, 1e-13])])
    t = torch.tensor(x, device="cuda")
    out = torch.empty((len(x), 2), dtype=torch.float32, device="cuda")
    assert lib.pairs_pow(t.data_ptr(), a, out.data_ptr(), len(x)) == 0
    got = out.cpu().numpy().astype(np.longdouble).sum(axis=-1)
    pairs = torch.empty((7, len(x), 2), dtype=torch.float32, device="cuda")  # (the power of the pair, which below 2^-97 is h alone)
    dbl = torch.empty(len(x), dtype=torch.float64, device="cuda")
    assert lib.pairs_check(t.data_ptr(), t.data_ptr(), t.data_ptr(), pairs.data_ptr(), dbl.data_ptr(), len(x)) == 0
    X, A = pairs[0].cpu().numpy().astype(np.longdouble).sum(axis=-1), np.longdouble(a)
    ref = X ** A
    ok = (ref > 1e-25) & (ref < 1e25)
    tol = np.longdouble(2.0) ** -44 * (1 + abs(A * np.log(X))) * ref
    assert np.all(abs(got - ref)[ok] <= tol[ok]), float(np.max((abs(got - ref) / tol)[ok]))


@pytest.mark.gpu
def test_power_of_bad_values(lib):
    import torch
    x = np.array([-1.0, np.nan, np.inf])
    t = torch.tensor(x, device="cuda")
    out = torch.empty((3, 2), dtype=torch.float32, device="cuda")
    assert lib.pairs_pow(t.data_ptr(), 0.76, out.data_ptr(), 3) == 0
    assert bool(torch.isnan(out.sum(dim=-1)).all())


@pytest.mark.gpu
def test_pair_to_double_on_the_integer_pipe(tmp_path):
    """The FP64 sum h + l of normalised pairs over the range of a stage's dt R, powers of two with a negative
    and a positive low part among them; the high part alone below 2^-66, NaN and infinity as NaN."""
    import torch
    out = str(tmp_path / "libpd.so")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "cuda", "pair_double_check.cu"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    lib.pair_double.argtypes = [ctypes.c_void_p] * 2 + [ctypes.c_int]
    rng = np.random.default_rng(5)
    n = 1 << 16
    h = (rng.choice([-1.0, 1.0], n) * rng.uniform(1.0, 2.0, n) * 2.0 ** rng.integers(-65, 100, n)).astype(np.float32)
    h[::4] = np.sign(h[::4]) * 2.0 ** np.floor(np.log2(np.abs(h[::4])))
    l = (rng.uniform(-0.5, 0.5, n) * np.spacing(np.abs(h))).astype(np.float32)
    l[::4] *= np.float32(0.5)  # (below a power of two the pair's low part is at most a quarter of its last place)
    l[1::8] = 0.0
    special = np.array([[0.0, 0.0], [-0.0, 0.0], [1e-25, 1e-33], [np.nan, 0.0], [np.inf, np.nan], [1.0, 2.0 ** -60]], dtype=np.float32)
    a = np.concatenate([np.stack([h, l], 1), special])
    t = torch.tensor(a, device="cuda")
    y = torch.empty(len(a), dtype=torch.float64, device="cuda")
    assert lib.pair_double(t.data_ptr(), y.data_ptr(), len(a)) == 0
    got = y.cpu().numpy()
    ref = h.astype(np.float64) + l.astype(np.float64)
    # l rounds to a multiple of the sum's last place, as the sum does (ties may differ)
    assert np.all(np.abs(got[:n] - ref) <= np.spacing(np.abs(ref)))
    assert np.mean(got[:n] == ref) > 0.99
    s = got[n:]
    assert s[0] == 0.0 and s[1] == 0.0 and s[2] == np.float64(np.float32(1e-25)) and np.isnan(s[3]) and np.isnan(s[4]) and s[5] == 1.0
