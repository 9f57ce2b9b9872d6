"""The line filter by itself: with a time step so small that the stages change nothing, one
synchronous step is the three filter passes, compared with a dense solve in extended precision."""
import numpy as np
import pytest

from paper_2506_03027_gb300 import cfs, inputs as I
from tests.gpu_util import ensure_built

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


def filter_axis(U, axis, p, alpha):
    """One pass along `axis` (counted from the end) in long double: every sub-domain line solved with
    its neighbours' values, f + (1 - 2 alpha)/1024 T^-1 delta^10 f."""
    n = U.shape[axis]
    base, rem = divmod(n, p)
    out = np.empty_like(U)
    o = 0
    for s in range(p):
        m = base + (s < rem)
        w = np.moveaxis(np.take(U, (np.arange(o - 5, o + m + 5)) % n, axis=axis), axis, -1)
        d = np.diff(w, 10, axis=-1)
        c = np.empty(m, dtype=np.longdouble)  # Thomas, in long double
        y = np.empty_like(d)
        piv = np.longdouble(1)
        for i in range(m):
            if i:
                piv = 1 - alpha * c[i - 1]
            c[i] = alpha / piv
            y[..., i] = (d[..., i] - (alpha * y[..., i - 1] if i else 0)) / piv
        for i in range(m - 2, -1, -1):
            y[..., i] = y[..., i] - c[i] * y[..., i + 1]
        r = w[..., 5:5 + m] + (1 - 2 * np.longdouble(alpha)) / 1024 * y
        np.moveaxis(out, axis, -1)[..., o:o + m] = r
        o += m
    return out


def rough_state(c, scale, seed):
    """Random point by point (the filter's largest increments), positive density and pressure."""
    rng = np.random.default_rng(seed)
    U = rng.uniform(-1.0, 1.0, size=(5, c.nz, c.ny, c.nx))
    U[0] = 2.0 + U[0]
    U[4] = 100.0 + U[4]
    return scale * U


# sub-domain lines of 5 points (the shortest), a ragged split, one longer than a warp's row of
# lanes, the longest block in one piece; values far from 1
@pytest.mark.parametrize("n,p,alpha,scale", [((10, 15, 10), (2, 3, 2), 0.499, 1.0), ((34, 20, 23), (4, 1, 2), 0.45, 1e-12),
                                            ((129, 12, 11), (1, 2, 1), 0.499, 1e12), ((13, 130, 97), (1, 1, 1), -0.3, 1.0)])
def test_filter_matches_extended_precision(n, p, alpha, scale):
    c = I.tgv_case(16, 1, "SA").replace(nx=n[0], ny=n[1], nz=n[2], px=p[0], py=p[1], pz=p[2], alpha_f=alpha, dt=1e-300)
    U0 = rough_state(c, scale, 7)
    s = cfs.Solver(c)
    s.set_schedule()
    s.set_state(U0)
    s.step(1)
    U = s.get_state()
    s.close()
    ref = U0.astype(np.longdouble)
    for axis in (-1, -2, -3):
        ref = filter_axis(ref, axis, p[-1 - axis], alpha)
    # per pass: half a unit in the last place of the sum, and at most as much again from the
    # fixed-point values and the sweeps, both of the variable's largest value
    for v in range(5):
        assert np.abs(U[v] - ref[v]).max() <= 3 * 2 * 2.0 ** -53 * np.abs(U0[v]).max(), v


def test_filter_leaves_vanishing_values_alone():
    """A variable that is zero but for the stages' dt R (below 1e-290) gets no increment."""
    c = I.tgv_case(16, 2, "SA").replace(dt=1e-300)
    U0 = rough_state(c, 1.0, 3)
    U0[3] = 0.0
    s = cfs.Solver(c)
    s.set_schedule()
    s.set_state(U0)
    s.step(1)
    U = s.get_state()
    s.close()
    assert np.all(np.abs(U[3]) < 1e-290) and np.all(np.isfinite(U))


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_nonfinite_value_reaches_its_lines(value):
    """A NaN or an infinity spreads over every line that sees it and is reported."""
    c = I.tgv_case(20, 2, "SA").replace(dt=1e-300)
    U0 = rough_state(c, 1.0, 5)
    U0[2, 9, 8, 7] = value
    s = cfs.Solver(c)
    s.set_schedule()
    s.set_state(U0)
    s.step(1)
    U = s.get_state()
    with pytest.raises(cfs.CfsError):
        s.diagnostics()
    s.close()
    assert np.all(np.isnan(U[2, 9, 8, :10]))


@pytest.mark.parametrize("filt", [False, True])
def test_memory_grows_with_the_line_not_its_square(filt, monkeypatch):
    """A context's tables (and the time to prepare them) are proportional to the longest line."""
    def total(n):
        sizes = []
        alloc = cfs.TorchAllocator._alloc
        with monkeypatch.context() as m:
            m.setattr(cfs.TorchAllocator, "_alloc", lambda self, b, user: (sizes.append(b), alloc(self, b, user))[1])
            s = cfs.Solver(I.vortex_case(32, 1).replace(nx=n, ny=8, filter=filt))
            s.close()
        return sum(sizes)
    a, b = total(340), total(680)
    assert b <= 2.0 * a, (a, b)


def one_pass(c, U0):
    s = cfs.Solver(c)
    s.set_schedule()
    s.set_state(U0)
    s.step(1)
    U = s.get_state()
    s.close()
    return U


def tailed_state(c, tail, seed):
    """Momenta of about 1 on the first third of every line along x and `tail` beyond it."""
    U = rough_state(c, 1.0, seed)
    U[1:4, :, :, c.nx // 3:] = tail(c.nx - c.nx // 3)
    return U


def reference(c, U0):
    ref = U0.astype(np.longdouble)
    for axis, p in ((-1, c.px), (-2, c.py), (-3, c.pz)):
        ref = filter_axis(ref, axis, p, c.alpha_f)
    return ref


# lines along x of 200 points in one piece and in two
@pytest.mark.parametrize("p", [1, 2])
def test_filter_of_opposite_and_vanishing_values(p):
    """-f filters to the opposite of f, and values far below the line's largest (of both signs, both
    zeros) take no rounding of the size of that one's."""
    c = I.tgv_case(16, 1, "SA").replace(nx=200, ny=12, nz=11, px=p, alpha_f=0.45, dt=1e-300)
    U0 = tailed_state(c, lambda n: 1e-30 * np.where(np.arange(n) % 3, -1.0, 1.0) * (np.arange(n) % 5 > 0), 9)
    U0[1:4][U0[1:4] == 0.0] *= -1.0
    V0 = U0.copy()
    V0[1:4] *= -1.0
    U, V = one_pass(c, U0), one_pass(c, V0)
    assert np.array_equal(U[1:4], -V[1:4])
    # the large values, and their rounding, reach into the rest of their line with (1 - sqrt(1 - 4
    # alpha^2)) / (2 alpha) = 0.63 per point: 1e-11 of their 2^-53 fifty-five points away
    e = np.abs(U - reference(c, U0))[1:4, :, :, 122:143].max()
    assert e <= 1e-24, e


# the small part in the middle of a sub-domain, over its end, and a step down and up again
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("scale", [1e-4, 1e-9, 1e-15])
def test_filter_of_small_values_beside_large_ones(p, scale):
    """Far from the large values the error is of the size of the rounding of the small ones."""
    rng = np.random.default_rng(21)
    c = I.tgv_case(16, 1, "SA").replace(nx=211, ny=12, nz=11, px=p, alpha_f=0.45, dt=1e-300)
    U0 = tailed_state(c, lambda n: scale * rng.uniform(-1.0, 1.0, n), 9)
    e = np.abs(one_pass(c, U0) - reference(c, U0))[1:4, :, :, 122:160]
    # per pass half a unit in the last place of the sum and the rounding of the fixed-point values, one
    # unit, seven binades below the place of which a line keeps its unit (the passes along y and z see
    # lines of one size).  Points within 18 of the large values take these's unit: of one unit there,
    # 0.63^33 = 2.1e-7 reaches fifty-one points away
    tol = (3 * 0.5 + 2 + 2.0 ** 7) * 2.0 ** -52 * scale + 2.1e-7 * 2.0 ** -52
    assert e.max() <= tol, (e.max(), tol)


def test_blocks_of_unequal_lines():
    """Blocks of long and short lines, whose launches overlap, in pieces and whole."""
    base = I.tgv_case(16, 1, "SA").replace(alpha_f=0.45, dt=1e-300)
    blocks = [base.replace(nx=n[0], ny=n[1], nz=n[2], px=p) for n, p in (((140, 10, 11), 1), ((12, 13, 10), 1), ((60, 11, 10), 2),
                                                                        ((100, 12, 10), 1), ((33, 10, 12), 3))]
    states = [rough_state(c, 1.0, 11 + k) for k, c in enumerate(blocks)]
    s = cfs.Solver(blocks[0], blocks=blocks)
    s.set_schedule()
    s.set_states(states)
    s.step(1)
    got = s.get_states()
    s.close()
    for c, U0, U in zip(blocks, states, got):
        ref = reference(c, U0)
        for v in range(5):
            assert np.abs(U[v] - ref[v]).max() <= 3 * 2 * 2.0 ** -53 * np.abs(U0[v]).max(), v
