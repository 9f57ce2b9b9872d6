"""The marching diagnostics kernel at the edges of its tiles, against plain numpy."""
import numpy as np
import pytest

from paper_2506_03027_gb300 import cfs, inputs as I
from tests.gpu_util import ensure_built

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


def reference(c, U):
    """K, enstrophy and the totals of a periodic Cartesian state."""
    vel = U[1:4] / U[0]

    def d(f, axis, h):
        a = np.roll(f, -1, axis) - np.roll(f, 1, axis)
        if c.order == 2:
            return a / (2 * h)
        return (8 * a - (np.roll(f, -2, axis) - np.roll(f, 2, axis))) / (12 * h)
    wx = d(vel[2], 1, c.dy) - d(vel[1], 0, c.dz)
    wy = d(vel[0], 0, c.dz) - d(vel[2], 2, c.dx)
    wz = d(vel[1], 2, c.dx) - d(vel[0], 1, c.dy)
    K = 0.5 * (U[0] * (vel ** 2).sum(axis=0)).mean()
    ens = 0.5 * (U[0] * (wx ** 2 + wy ** 2 + wz ** 2)).mean()
    return np.array([K, ens, *(U.reshape(5, -1).sum(axis=1) * c.dx * c.dy * c.dz)])


def state(c, seed, scale=1.0):
    rng = np.random.default_rng(seed)
    U = rng.uniform(-1.0, 1.0, size=(5, c.nz, c.ny, c.nx))
    U[0] = 1.5 + 0.3 * U[0]
    U[4] += 50.0
    return U * scale


def static(c, U):
    import torch
    t = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    out = torch.zeros(8, dtype=torch.float64, device="cuda")
    cfs.cfs_diagnostics_static(t.data_ptr(), c.nx, c.ny, c.nz, (c.dx, c.dy, c.dz), c.order, out.data_ptr(),
                               torch.cuda.current_stream().cuda_stream)
    return out.cpu().numpy()


# one tile and less, one point more than a tile, a chunk of planes and one more, stencils that wrap
# onto themselves, unequal spacings; values outside the range of the pairs (taken in FP64)
@pytest.mark.parametrize("n", [(32, 8, 8), (33, 9, 9), (5, 3, 2), (70, 17, 25), (1, 40, 12), (129, 2, 3)])
@pytest.mark.parametrize("order,scale", [(4, 1.0), (2, 1.0), (4, 1e25)])
def test_tiles(n, order, scale):
    c = I.tgv_case(16, 1, "SA").replace(nx=n[0], ny=n[1], nz=n[2], lx=1.3, ly=2.0, lz=0.7, order=order)
    U = state(c, 3, scale)
    ref = reference(c, U)
    mag = np.abs(U).reshape(5, -1).sum(axis=1) * c.dx * c.dy * c.dz
    got = static(c, U)
    assert np.all(np.abs(got[:2] - ref[:2]) <= 1e-13 * np.abs(ref[:2]))
    assert np.all(np.abs(got[2:7] - ref[2:7]) <= 1e-13 * mag) and got[7] == 0.0


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_nonfinite_value_is_flagged(value):
    c = I.tgv_case(16, 1, "SA").replace(nx=40, ny=20, nz=18)
    U = state(c, 4)
    U[4, 17, 19, 39] = value
    got = static(c, U)
    assert got[7] == 1.0
    s = cfs.Solver(c)
    s.set_schedule()
    s.set_state(U)
    with pytest.raises(cfs.CfsError) as e:
        s.diagnostics()
    s.close()
    assert e.value.status == cfs.CFS_ENAN


# products of values inside the pairs' range that leave it, above (velocities of 2^65) and below (of 1e-25
# and 1e-15), and a spacing that leaves it
@pytest.mark.parametrize("rho,vel,box", [(2.0 ** -30, 2.0 ** 65, 1.0), (2.0 ** 20, 2.0 ** -85, 1.0), (1.0, 1e-25, 1.0), (1.0, 1e-15, 1.0),
                                         (1.0, 1.0, 1e25), (1.0, 1.0, 1e-25)])
def test_products_outside_the_pairs_range(rho, vel, box):
    c = I.tgv_case(16, 1, "SA").replace(nx=70, ny=60, nz=64, lx=1.3 * box, ly=2.0 * box, lz=0.7 * box)
    U = state(c, 3)
    U[0] *= rho
    U[1:4] *= rho * vel
    ref = reference(c, U)
    got = static(c, U)
    # (pairs: 2^-48 of the velocities, whose differences are of their size)
    assert np.all(np.abs(got[:2] - ref[:2]) <= 1e-13 * np.abs(ref[:2])), (got[:2], ref[:2])
    assert got[7] == 0.0


def test_mixed_scales():
    """Slabs of slow fluid beside fast ones, and fluid at rest, keep the totals."""
    c = I.tgv_case(16, 1, "SA").replace(nx=70, ny=60, nz=64)
    U = state(c, 3)
    U[1:4, 10:50] *= 1e-20
    U[1:4, 55:] = 0.0
    ref, got = reference(c, U), static(c, U)
    assert np.all(np.abs(got[:2] - ref[:2]) <= 1e-13 * np.abs(ref[:2])) and got[7] == 0.0


# shapes that the marching kernel takes (a column and a row more than its tiles, a last chunk of fewer planes),
# and slender and small ones that the kernel by points does
@pytest.mark.parametrize("n", [(65, 57, 66), (64, 64, 64), (96, 65, 53), (129, 41, 50), (3, 5, 4000), (2, 300, 40), (33, 32, 32)])
@pytest.mark.parametrize("order,scale", [(4, 1.0), (2, 1.0), (4, 1e25)])
def test_shapes(n, order, scale):
    test_tiles(n, order, scale)
