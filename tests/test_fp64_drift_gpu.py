"""The velocity of a fast, nearly steady flow over 200 FP64 steps, against the same steps
in extended precision (numpy's long double, with the quadrature constants as doubles).

A site whose state hardly changes repeats its rounding errors every step.  Its velocity is
rounded once a step (u = c j / rho + g / 2 as one fused operation), by at most U 2^-53, so
200 steps move it by at most 200 U 2^-53; with a second rounding (of the product) they may
move it by twice that, and did, by 1.5 times.
"""
import numpy as np
import pytest

import paper_2302_04741_gb300 as lbm
from helpers import workload

pytestmark = pytest.mark.gpu

NY, U, MU, G, STEPS = 150, 1.2, 0.15, (1e-4, -1e-4), 200


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2302_04741_gb300 import build
    build.build()


class Column:
    """A periodic D2Q37 flow that is uniform in x: deviations d[37, NY]."""

    def __init__(self, real):
        _, Q, c, e, w = lbm.lbm_lattice_info(lbm.LBM_D2Q37)
        self.e, self.real = e[:, :2], real
        self.c, self.w = real(c), w.astype(real)[:, None]
        self.ex, self.ey = (e[:, a].astype(real)[:, None] for a in (0, 1))
        self.g = np.array(G, real)[:, None]

    def pull(self, d):
        return np.stack([np.roll(d[i], self.e[i, 1]) for i in range(37)])

    def moments(self, d):
        e2 = self.ex * self.ex + self.ey * self.ey
        m0 = d.sum(0)
        rho = 1 + m0
        ut = self.c * np.stack([(self.ex * d).sum(0), (self.ey * d).sum(0)]) / rho
        Th = ((self.c * self.c * (e2 * d).sum(0) - 2 * m0) / rho - (ut * ut).sum(0)) / 2 + (self.g * self.g).sum(0) / 8
        return m0, rho, ut + self.g / 2, Th

    def shape(self, u, Th):
        """(t, s, f0 / (w rho) - 1, F / (w rho)) for every direction."""
        c, ex, ey = self.c, self.ex, self.ey
        t, s, X2 = c * (ex * u[0] + ey * u[1]), c * (ex * self.g[0] + ey * self.g[1]), c * c * (ex * ex + ey * ey)
        u2, gu = (u * u).sum(0), (self.g * u).sum(0)
        Z = Th * (X2 - 4) - u2
        h = t + (t * t - u2 + Th * (X2 - 2)) / 2 + t * (t * t + 3 * Z) / 6
        h = h + (t ** 4 + 6 * t * t * (Th * (X2 - 6) - u2) + 3 * u2 * u2 - 6 * Th * u2 * (X2 - 4)
                 + 3 * Th * Th * (X2 * X2 - 8 * X2 + 8)) / 24
        return h, s * (1 + t + (t * t + Z) / 2) - gu * (1 + t)

    def step(self, d):
        d = self.pull(d)
        m0, rho, u, Th = self.moments(d)
        om = 1 / (self.real(MU) / (rho * (1 + Th)) + self.real(0.5))
        h, F = self.shape(u, Th)
        return d - om * (d - self.w * (m0 + rho * h)) + (1 - om / 2) * self.w * rho * F


@pytest.fixture(scope="module")
def flow():
    """Stored populations of the first state, and the velocity after STEPS steps."""
    x = Column(np.longdouble)
    y = 2 * np.pi * (np.arange(NY) + 0.25) / NY
    u = np.array([U * np.sin(y), 0.05 * np.cos(y)], np.longdouble)
    Th, rho = np.longdouble(0.1) * np.cos(y), 1 + np.longdouble(0.02) * np.sin(2 * y)
    h, _ = x.shape(u, Th)
    f = (x.w * (rho + rho * h)).astype(np.float64)
    d = f.astype(np.longdouble) - x.w
    for _ in range(STEPS):
        d = x.step(d)
    return f, x.moments(x.pull(d))[2]


# 8 lanes a site, 2 lanes, one thread
@pytest.mark.parametrize("nx", [3, 40, 70])
def test_the_velocity_is_rounded_once_a_step(flow, nx):
    f, want = flow
    w = workload(0, (nx, NY, 1), g={"kind": lbm.LBM_G_UNIFORM, "g0": (*G, 0.0)})
    w["mu"] = MU
    sim = lbm.Sim(w).init()
    sim.set_state(np.repeat(f[:, :, None], nx, 2).reshape(37, nx * NY))
    sim.step(STEPS)
    x = Column(np.longdouble)
    d = np.asarray(sim.get_state()).reshape(37, NY, nx)[:, :, nx // 2].astype(np.longdouble) - x.w
    got = x.moments(x.pull(d))[2]
    assert float(np.abs(got - want).max()) <= STEPS * U * 2.0 ** -53
