"""The specialised stage kernels at the edges of their tiles and forms, against the oracle: the one-launch
stage of two-dimensional inviscid runs, the compact scheme's lines, the FP32 form's halo store with the
latest delayed level, and the halo network's kernels at batches around their tiles."""
import numpy as np
import pytest

from oracle import mlp as omlp
from oracle import oracle as orc
from paper_2506_03027_gb300 import cfs
from paper_2506_03027_gb300 import inputs as I
from paper_2506_03027_gb300 import learned as L

from gpu_util import PARITY_TOL, ensure_built, gpu_run, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()


def smooth_2d(c, seed):
    """A smooth periodic state that is not symmetric in x and y and moves in z too."""
    rng = np.random.default_rng(seed)
    y, x = np.meshgrid(2 * np.pi * np.arange(c.ny) / c.ny, 2 * np.pi * np.arange(c.nx) / c.nx, indexing="ij")
    ph = rng.uniform(0, 2 * np.pi, 5)
    rho = 1 + 0.1 * np.sin(x + 2 * y + ph[0])
    vel = [0.3 * np.sin(2 * x - y + ph[1]), 0.2 * np.cos(x + y + ph[2]), 0.25 * np.sin(x - y + ph[3])]
    p = (1 + 0.1 * np.cos(2 * x + y + ph[4])) / (c.gamma * c.mach ** 2)
    U = np.zeros((5, 1, c.ny, c.nx))
    U[0, 0] = rho
    for k in range(3):
        U[1 + k, 0] = rho * vel[k]
    U[4, 0] = p / (c.gamma - 1) + 0.5 * rho * sum(v * v for v in vel)
    return U


# sub-domains smaller than a tile, of one tile exactly, one point more, ragged ones, and a grid
# that takes the large tiles (more than 2736 small ones at fourth order); unequal spacings
@pytest.mark.parametrize("n,p", [((8, 8), (1, 1)), ((9, 17), (1, 2)), ((35, 22), (3, 2)), ((64, 16), (1, 1)),
                                 ((501, 377), (5, 4))])
@pytest.mark.parametrize("order,algo,at", [(4, "SA", True), (2, "CAA", True), (4, "SAA", True), (4, "SAA", False)])
def test_two_dimensional_inviscid_stage(n, p, order, algo, at):
    c = I.vortex_case(32, 1, order=order).replace(nx=n[0], ny=n[1], px=p[0], py=p[1], lx=10.0, ly=7.0, algo=algo, at=at, kmax=2)
    U0 = smooth_2d(c, 5)
    c = c.replace(dt=I.cfl_dt(c, U0, 0.2))
    nst = 10
    d = I.saa_delays(c, nst) if algo == "SAA" else None
    Ug, _ = gpu_run(c, U0, nst, delays=d)
    e = rel_l2(Ug, orc.run(c, U0, nst, delays=d))
    assert np.all(np.isfinite(Ug)) and np.all(e <= PARITY_TOL), e


# a line per CTA slot and less, one more than the 64 of a CTA, long lines, different splits per axis
@pytest.mark.parametrize("n,p", [((16, 8, 8), (1, 1, 1)), ((13, 21, 9), (1, 2, 1)), ((40, 33, 26), (1, 3, 2))])
def test_compact_lines(n, p):
    c = I.tgv_case(16, 1, "CAA", viscous=False, compact=1).replace(nx=n[0], ny=n[1], nz=n[2], px=p[0], py=p[1], pz=p[2])
    U0 = I.tgv_state(c)
    c = c.replace(dt=I.cfl_dt(c, U0, 0.25))
    Ug, _ = gpu_run(c, U0, 10)
    e = rel_l2(Ug, orc.run(c, U0, 10))
    assert np.all(np.isfinite(Ug)) and np.all(e <= PARITY_TOL), e


# sub-domains of 16^3 and 32^3 (the halo store and the sub-domain filter's halos in one launch)
@pytest.mark.parametrize("n", [32, 64])
@pytest.mark.parametrize("algo", ["CAA", "SAA"])
def test_fp32_halo_store_latest_level(n, algo):
    c = I.tgv_case(n, 2, algo, at=False, kmax=2)
    U0 = I.tgv_state(c)
    c = c.replace(dt=I.cfl_dt(c, U0, 0.1))
    d = I.saa_delays(c, 10) if algo == "SAA" else None
    Ug, _ = gpu_run(c, U0, 10, delays=d, precision=1)
    e = rel_l2(Ug, orc.run(c, U0, 10, delays=d))
    assert np.all(np.isfinite(Ug)) and np.all(e < 1e-6), e


# one sample, odd batches, one more and one less than the tiles, inputs and workspace at an offset
@pytest.mark.parametrize("n", [1, 3, 31, 33, 127, 129, 257, 1021])
@pytest.mark.parametrize("offset", [0, 1])
def test_network_batches(n, offset):
    import torch
    rng = np.random.default_rng(n)
    p = L.init_params(4)
    x = rng.standard_normal((n + offset, omlp.NIN)).astype(np.float32)
    bits = ((x.view(np.uint32) + 0x7FFF + ((x.view(np.uint32) >> 16) & 1)) >> 16).astype(np.uint32)
    xb = (bits << 16).view(np.float32).astype(np.float64)[offset:]
    T = rng.standard_normal((n, omlp.NOUT)).astype(np.float32)
    pt = torch.from_numpy(p).cuda()
    xt = torch.from_numpy(bits.astype(np.uint16).view(np.int16)).cuda()[offset:]
    tt = torch.from_numpy(T).cuda()
    g, loss = torch.zeros_like(pt), torch.zeros(1, device="cuda")
    ws = torch.empty(cfs.cfs_mlp_workspace_bytes(n) // 4 + 1 + offset, device="cuda")[offset:]
    cfs.cfs_mlp_grad(pt.data_ptr(), xt.data_ptr(), tt.data_ptr(), n, ws.data_ptr(), g.data_ptr(), loss.data_ptr())
    lref, gref = omlp.loss_and_grad(p.astype(np.float64), xb, T.astype(np.float64))
    gg = g.cpu().numpy().astype(np.float64)
    assert abs(loss.item() - lref) <= 1e-5 * lref
    assert np.linalg.norm(gg - gref) <= 1e-5 * np.linalg.norm(gref)
    ref = omlp.forward(p.astype(np.float64), xb)[0]
    y = L.predict(p, xt).cpu().numpy().astype(np.float64)
    assert np.abs(y - ref).max() <= 2e-5 * max(1.0, np.abs(ref).max())


# no memory for the halo values of all stages: the FP64 kernels take the run
@pytest.mark.parametrize("kind", ["viscous", "power_law", "euler", "compact"])
def test_run_without_room_for_the_halo_values(kind, monkeypatch):
    kw = {"viscous": {}, "power_law": {"visc_law": 1}, "euler": {"viscous": False}, "compact": {"viscous": False, "compact": 1}}[kind]
    c = I.tgv_case(26, 2, "CAA", **kw)
    U0 = I.tgv_state(c)
    c = c.replace(dt=I.cfl_dt(c, U0, 0.25))
    G, r = (4, 2) if kind != "euler" else (2, 2)
    w = 13
    entries = c.nsub * 6 * w * w * G + (c.nsub * 12 * r * r * w if c.viscous else 0)
    refused = []
    alloc = cfs.TorchAllocator._alloc

    def without(self, nbytes, user):
        if nbytes == 40 * c.stages * entries:
            refused.append(nbytes)
            return None
        return alloc(self, nbytes, user)
    monkeypatch.setattr(cfs.TorchAllocator, "_alloc", without)
    Ug, _ = gpu_run(c, U0, 10)
    assert len(refused) == 1
    e = rel_l2(Ug, orc.run(c, U0, 10))
    assert np.all(np.isfinite(Ug)) and np.all(e <= PARITY_TOL), e


def limited(monkeypatch, allowed):
    """The allocator refuses what `allowed(bytes, bytes in use)` does not grant; the refused sizes."""
    refused = []
    alloc, free = cfs.TorchAllocator._alloc, cfs.TorchAllocator._free
    held = {}

    def get(self, nbytes, user):
        if not allowed(nbytes, sum(held.values())):
            refused.append(nbytes)
            return None
        p = alloc(self, nbytes, user)
        held[p] = nbytes
        return p

    def put(self, ptr, user):
        held.pop(ptr, None)
        free(self, ptr, user)
    monkeypatch.setattr(cfs.TorchAllocator, "_alloc", get)
    monkeypatch.setattr(cfs.TorchAllocator, "_free", put)
    return refused


def advance(c, precision=0, graph=False, learned=False, steps=9):
    import torch
    U0 = I.tgv_state(c)
    s = cfs.Solver(c, precision=precision, graph=graph, stream=torch.cuda.Stream())
    s.set_schedule(delays=I.saa_delays(c, steps) if c.algo == "SAA" else None)
    if learned:
        cfs.cfs_set_halo_model(s.ctx, L.init_params(4),
                               np.array([3e3, 2e3, 2e3, 2e3, 1e3, 4e2, 3e2, 3e2, 3e2, 2e2, 1e7, 1e6, 1e6, 1e6, 5e5]))
    s.set_state(U0)
    s.step(steps)
    U = s.get_state()
    s.close()
    return U


FORMS = {"viscous": (26, {}, {}), "power_law_graph": (26, {"visc_law": 1}, {"graph": True}), "euler": (26, {"viscous": False}, {}),
         "compact": (26, {"viscous": False, "compact": 1}, {}), "latest_level": (26, {"at": False}, {}), "order2": (26, {"order": 2}, {}),
         "fp32": (26, {}, {"precision": 1}), "fp32_cubes": (32, {}, {"precision": 1}), "fp32_cubes_graph": (32, {}, {"precision": 1, "graph": True}),
         "fp32_latest_level": (32, {"at": False}, {"precision": 1})}


# where there is no memory for the halo values of all stages, those of one at a time give the same bits
@pytest.mark.parametrize("form", list(FORMS))
def test_same_values_without_room_for_all_stages(form, monkeypatch):
    n, kw, run = FORMS[form]
    c = I.tgv_case(n, 2, "SAA", kmax=2, **kw)
    c = c.replace(dt=I.cfl_dt(c, I.tgv_state(c), 0.1))
    sizes = []
    with monkeypatch.context() as m:
        limited(m, lambda b, used: sizes.append(b) or True)
        full = advance(c, **run)
    w = n // 2
    if run.get("precision"):
        store = 4 * 8 * c.stages * c.nsub * (w + 8) ** 3
    else:
        G, r = (4, 2) if c.compact else ((2 * (c.order // 2), c.order // 2) if c.viscous else (2, 2))
        store = 40 * c.stages * (c.nsub * 6 * w * w * G + (c.nsub * 12 * r * r * w if c.viscous else 0))
    assert sizes.count(store) == 1
    with monkeypatch.context() as m:
        refused = limited(m, lambda b, used: b != store)
        one = advance(c, **run)
    assert refused == [store]
    assert np.all(np.isfinite(full)) and np.array_equal(full, one)


# the store gives way to what is allocated after it, here the halo network's buffers
@pytest.mark.parametrize("precision", [0, 1])
def test_store_of_all_stages_gives_way(precision, monkeypatch):
    c = I.tgv_case(32, 2, "SAA", kmax=2)
    c = c.replace(dt=I.cfl_dt(c, I.tgv_state(c), 0.1))
    peak = []
    with monkeypatch.context() as m:
        limited(m, lambda b, used: peak.append(used + b) or True)
        full = advance(c, precision=precision, learned=True)
    with monkeypatch.context() as m:
        refused = limited(m, lambda b, used: used + b < max(peak))
        one = advance(c, precision=precision, learned=True)
    assert len(refused) == 1
    assert np.all(np.isfinite(full)) and np.array_equal(full, one)


# the launches of a step: large tiles where the sub-domains' rows fill them (the second size ragged), three kernels
# per stage where they do not, small tiles on small grids of either
@pytest.mark.parametrize("n,p,order,launches", [((512, 448), (8, 7), 4, 5), ((510, 443), (8, 7), 4, 5), ((512, 448), (8, 7), 2, 2),
                                                ((528, 528), (16, 16), 4, 15), ((528, 528), (16, 16), 2, 6), ((99, 99), (3, 3), 4, 5),
                                                ((99, 99), (3, 3), 2, 2)])
def test_two_dimensional_inviscid_route(n, p, order, launches):
    c = I.vortex_case(32, 1, order=order).replace(nx=n[0], ny=n[1], px=p[0], py=p[1], lx=10.0, ly=7.0)
    U0 = smooth_2d(c, 5)
    c = c.replace(dt=I.cfl_dt(c, U0, 0.2))
    s = cfs.Solver(c)
    s.set_schedule()
    s.set_state(U0)
    s.step(1)
    assert s.launches() == launches
    U = s.get_state()
    s.close()
    assert np.all(rel_l2(U, orc.run(c, U0, 1)) <= PARITY_TOL)


# more sub-domains than the second dimension of a grid counts
@pytest.mark.parametrize("n", [16, 32])
def test_halo_store_of_many_subdomains(n, tmp_path):
    import ctypes
    import os
    import subprocess
    from paper_2506_03027_gb300 import build as B
    here = os.path.dirname(os.path.abspath(__file__))
    out = str(tmp_path / "liblaunch.so")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", B.CSRC,
                    os.path.join(here, "cuda", "launch_check.cu"), B.LIB, "-Xlinker", "-rpath=" + os.path.dirname(B.LIB), "-o", out], check=True)
    assert ctypes.CDLL(out).halo_block_launch(70000, n) == 0


# a NaN or an infinity in another component reaches the z momentum though that is zero
@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("component", [0, 1, 2])
@pytest.mark.parametrize("n", [(35, 22), (510, 443)])
def test_nonfinite_value_reaches_the_zero_z_momentum(n, component, value):
    c = I.vortex_case(32, 1).replace(nx=n[0], ny=n[1], px=max(1, n[0] // 60), py=max(1, n[1] // 60), lx=10.0, ly=7.0, dt=1e-4)
    U0 = smooth_2d(c, 5)
    U0[3] = 0.0
    U0[component, 0, 9, 17] = value
    Ug, _ = gpu_run(c, U0, 1)
    ref = orc.run(c, U0, 1)
    assert not np.all(np.isfinite(ref[3]))
    assert np.array_equal(np.isfinite(Ug[3]), np.isfinite(ref[3]))
