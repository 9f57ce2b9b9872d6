"""One synchronous step of the three-dimensional solver in extended precision (numpy's long double),
written from the method's definition, for tests that resolve errors below the rounding of FP64."""
import numpy as np

from oracle import oracle as orc

LD = np.longdouble


def _diff(f, axis, h, order):
    d1 = np.roll(f, -1, axis) - np.roll(f, 1, axis)
    if order == 2:
        return d1 / (2 * h)
    return (8 * d1 - (np.roll(f, -2, axis) - np.roll(f, 2, axis))) / (12 * h)


def _compact(f, axis, h):
    """Sixth-order compact derivative of periodic lines of one sub-domain, closed by the explicit
    sixth-order difference at the point beyond each end."""
    f = np.moveaxis(f, axis, -1)
    n = f.shape[-1]

    def at(o):
        return f[..., (np.arange(-1, n + 1) + o) % n]
    ex = (45 * (at(1) - at(-1)) - 9 * (at(2) - at(-2)) + (at(3) - at(-3))) / (60 * h)
    rhs = (LD(14) / 9 * (at(1) - at(-1)) / (2 * h) + LD(1) / 9 * (at(2) - at(-2)) / (4 * h))[..., 1:-1].copy()
    rhs[..., 0] -= ex[..., 0] / 3
    rhs[..., -1] -= ex[..., -1] / 3
    c, piv = np.zeros(n, LD), LD(1)
    for i in range(n):
        if i:
            piv = 1 - c[i - 1] / 3
            rhs[..., i] -= rhs[..., i - 1] / 3
        c[i] = 1 / (3 * piv)
        rhs[..., i] /= piv
    for i in range(n - 2, -1, -1):
        rhs[..., i] -= c[i] * rhs[..., i + 1]
    return np.moveaxis(rhs, -1, axis)


def rhs(c, U):
    """R(U) of a periodic Cartesian block in one sub-domain (App. A), long double."""
    lx = (LD(c.dx), LD(c.dy), LD(c.dz))
    gamma, M, Re, Pr = (LD(x) for x in (c.gamma, c.mach, c.re, c.pr))
    rho = U[0]
    u = [U[1 + a] / rho for a in range(3)]
    p = (gamma - 1) * (U[4] - (U[1] * u[0] + U[2] * u[1] + U[3] * u[2]) / 2)

    def d(f, a):
        return _diff(f, 2 - a, lx[a], c.order)
    if c.viscous:
        T = gamma * M * M * p / rho
        mu = T ** LD(c.visc_exp) if c.visc_law == 1 else 1
        g = [[d(f, a) for a in range(3)] for f in u + [T]]
        div = g[0][0] + g[1][1] + g[2][2]
        kappa = 1 / ((gamma - 1) * Pr * M * M)
    R = 0
    for a in range(3):
        F = [-U[1 + a]] + [-U[1 + i] * u[a] for i in range(3)] + [-(U[4] + p) * u[a]]
        F[1 + a] = F[1 + a] - p
        if c.viscous:
            tau = [mu * (g[a][i] + g[i][a]) - (2 * mu * div / 3 if i == a else 0) for i in range(3)]
            for i in range(3):
                F[1 + i] = F[1 + i] + tau[i] / Re
            F[4] = F[4] + (sum(u[i] * tau[i] for i in range(3)) + kappa * mu * g[3][a]) / Re
        R = R + np.stack([_compact(f, 2 - a, lx[a]) if c.compact else d(f, a) for f in F])
    return R


def step(c, U0):
    """The state after one synchronous step without the filter, long double."""
    A, B = orc.lserk(c.order)
    U = U0.astype(LD)
    Q = np.zeros_like(U)
    for m in range(c.stages):
        Q = LD(A[m]) * Q + LD(c.dt) * rhs(c, U)
        U = U + LD(B[m]) * Q
    return U
