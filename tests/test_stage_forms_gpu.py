"""The FP64 form's three-dimensional stage over its forms, against the oracle, with the filter (right-hand side
on pairs of floats) and without it (FP64 kernels): orders, periodic deformed and connected grids, power law,
latest delayed level, inviscid, learned halo, partition."""
import numpy as np
import pytest

import test_partition_gpu as partition
from oracle import oracle as orc
from paper_2506_03027_gb300 import cfs
from paper_2506_03027_gb300 import inputs as I
from paper_2506_03027_gb300 import learned as L

from gpu_util import PARITY_TOL, ensure_built, gpu_run, rel_l2
from test_blocks_gpu import cgrid, check_blocks, run_mb, sub_delays

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()


FORMS = {"viscous": {}, "order2": {"order": 2}, "power_law": {"visc_law": 1}, "latest_level": {"at": False}, "euler": {"viscous": False},
         "deformed": {"curv": 0.2}, "deformed_order2": {"curv": 0.2, "order": 2}, "deformed_power_law": {"curv": 0.2, "visc_law": 1},
         "deformed_power_law_order2": {"curv": 0.2, "visc_law": 1, "order": 2}, "deformed_latest_level": {"curv": 0.2, "at": False},
         "deformed_euler": {"curv": 0.2, "viscous": False}}


@pytest.mark.parametrize("filt", [True, False])
@pytest.mark.parametrize("algo", ["SA", "SAA"])
@pytest.mark.parametrize("form", list(FORMS))
def test_periodic_block(form, algo, filt):
    c = I.tgv_case(22, 2, algo, filter=filt, **FORMS[form]).replace(px=3, kmax=2)
    U0 = I.tgv_state(c)
    c = c.replace(dt=I.cfl_dt(c, U0, 0.1))
    d = I.saa_delays(c, 12) if algo == "SAA" else None
    Ug, _ = gpu_run(c, U0, 12, delays=d)
    e = rel_l2(Ug, orc.run(c, U0, 12, delays=d))
    assert np.all(np.isfinite(Ug)) and np.all(e <= PARITY_TOL), e


@pytest.mark.parametrize("filt,at", [(False, True), (True, False), (False, False)])
def test_connected_grid(filt, at):
    mb, U0 = cgrid("SAA")
    mb = mb.replace_all(filter=filt, at=at)
    d = sub_delays(mb, 12)
    check_blocks(run_mb(mb, U0, 12, delays=d), orc.run(mb, U0, 12, delays=d))


def test_wall_channel_without_the_filter():
    c = I.tgv_case(20, 2, "SAA", kmax=2, filter=False).replace(ny=21, py=3, ly=2.0)
    U = I.tgv_state(c)
    U[1:4, :, 0, :] = 0.0
    U[1:4, :, -1, :] = 0.0
    c = c.replace(dt=I.cfl_dt(c, U, 0.1))
    mb = I.wall_channel(c)
    d = I.saa_delays(c, 16)
    Ug = run_mb(mb, [U], 16, delays=d)
    check_blocks(Ug, orc.run(mb, [U], 16, delays=d))
    assert np.all(Ug[0][1:4, :, 0, :] == 0.0) and np.all(Ug[0][1:4, :, -1, :] == 0.0)


SCALES = np.array([3e3, 2e3, 2e3, 2e3, 1e3, 4e2, 3e2, 3e2, 3e2, 2e2, 1e7, 1e6, 1e6, 1e6, 5e5])


def learned_run(c, d, params):
    s = cfs.Solver(c, max_delay=4)
    s.set_schedule(delays=d)
    if params is not None:
        cfs.cfs_set_halo_model(s.ctx, params, SCALES)
    s.set_state(I.tgv_state(c))
    s.step(12)
    U = s.get_state()
    s.close()
    assert np.all(np.isfinite(U))
    return U


def learned_case(**kw):
    c = I.tgv_case(24, 2, "SAA", kmax=4, **kw)
    return c.replace(dt=I.cfl_dt(c, I.tgv_state(c), 0.05))


@pytest.mark.parametrize("kw", [{"filter": False}, {"curv": 0.2, "filter": True}])
def test_learned_halo(kw):
    c = learned_case(**kw)
    d = I.saa_delays(c, 12)
    params = L.init_params(7)
    # (the bound of the solver's own comparison: the network's BF16 inputs round on either side)
    e = rel_l2(learned_run(c, d, params), orc.run(c, I.tgv_state(c), 12, delays=d, model=(params, SCALES)))
    assert np.all(e <= 1e-11), e


def test_learned_halo_of_the_compact_scheme():
    """The FP64 kernels (no filter) against the pairs (a filter that does nothing, alpha_f next to 1/2)."""
    c = learned_case(viscous=False, compact=1, filter=False)
    d = I.saa_delays(c, 12)
    params = L.init_params(7)
    U = learned_run(c, d, params)
    e = rel_l2(learned_run(c.replace(filter=True, alpha_f=float(np.nextafter(0.5, 0))), d, params), U)
    assert np.all(e <= 1e-11), e
    assert rel_l2(U, learned_run(c, d, None)).max() > 100 * e.max()  # the network really changed the run


def rank_without_filter(*args):
    filtered = partition._case
    partition._case = lambda name: filtered(name).replace(filter=False)
    partition._rank(*args)


@pytest.mark.parametrize("name,starts", [("SA", [0, 32, 64]), ("SAA", [0, 40, 64])])
def test_two_processes_without_the_filter(name, starts):
    import torch.multiprocessing as mp
    mctx = mp.get_context("spawn")
    with mctx.Manager() as mgr:
        out = mgr.dict()
        port = partition._free_port()
        procs = [mctx.Process(target=rank_without_filter, args=(r, 2, port, name, starts, 10, out)) for r in range(2)]
        for p in procs:
            p.start()
        for p in procs:
            p.join(timeout=600)
        for p in procs:
            if p.is_alive():
                p.terminate()
                p.join(timeout=30)
        assert all(p.exitcode == 0 for p in procs), [p.exitcode for p in procs]
        res = dict(out)
    assert all(res[r][0] for r in range(2)), [res[r][1] for r in range(2)]
