"""The FP64 collision (IEEE double and float-float) on states far from rest.

The collision evaluates equilibrium and force by parity classes of the
directions, so every coefficient of every order matters; amplitudes of 0.3 in
velocity and 0.2 in temperature and density make each of them visible.

Tolerance per population, absolute, after three steps: some 40 rounded
operations on terms below 0.3 a step give 40 x 3 x 0.3 x 2^-53 = 4e-15 in
double; the float-float arithmetic carries 48 bits, 32 times that.
"""
import os

import numpy as np
import pytest

import oracle
import paper_2302_04741_gb300 as lbm
from paper_2302_04741_gb300 import workloads as W
from helpers import oracle_sim, perm_to_oracle, smooth_state, workload

pytestmark = pytest.mark.gpu

TOL = {lbm.LBM_ARITH_DOUBLE: 5e-15, lbm.LBM_ARITH_FLOAT_PAIR: 1.6e-13}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2302_04741_gb300 import build
    build.build()
    oracle.set_threads(os.cpu_count() or 1)


# one row wider than a warp and its wrap, rows at and between walls; the D2Q37
# grids also span the step's lanes per site (8 up to 608 sites, 2 up to 9,728,
# then one thread per site), with sites that do not fill the last warp
GRIDS = [(0, (3, 150, 1)), (0, (13, 7, 1)), (0, (71, 13, 1)), (0, (101, 96, 1)), (0, (101, 99, 1)), (1, (71, 7, 9))]


@pytest.mark.parametrize("arith", [0, 1], ids=["double", "pair"])
@pytest.mark.parametrize("order,sigma", [(0, False), (1, False), (2, False), (2, True)])
@pytest.mark.parametrize("wall", [0, 1, 2], ids=["periodic", "bounce", "thermal"])
@pytest.mark.parametrize("lat,shape", GRIDS, ids=["x".join(map(str, s)) for _, s in GRIDS])
def test_strong_flow(lat, shape, wall, order, sigma, arith):
    D = W.dims(lat)
    g = {"kind": W.G_UNIFORM, "g0": (0.03, -0.05, 0.02 if D == 3 else 0.0)}
    bc, T_lo, T_hi = [0, 0, 0], [1.0] * 3, [1.0] * 3
    bc[D - 1], T_lo[D - 1], T_hi[D - 1] = wall, 1.15, 0.9
    w = workload(lat, shape, tau=0.7, g=g, force_order=order, bc=tuple(bc))
    w["T_lo"], w["T_hi"] = tuple(T_lo), tuple(T_hi)
    w["rho"], w["u"], w["T"] = smooth_state(lat, shape, 11, amp_u=0.3, amp_T=0.2, amp_rho=0.2)
    w["include_sigma"], w["fp64_arith"] = sigma, arith
    sim, ref = lbm.Sim(w).init(), oracle_sim(w)
    sim.step(3)
    ref.step(3)
    far = np.abs(sim.populations() - ref.pulled()[perm_to_oracle(lat)])
    assert far.max() < TOL[arith]


@pytest.mark.parametrize("lat,shape", GRIDS[:5], ids=["x".join(map(str, s)) for _, s in GRIDS[:5]])
@pytest.mark.parametrize("force", ["mu", "sine", "field"])
@pytest.mark.parametrize("wall", [0, 2], ids=["periodic", "thermal"])
def test_forces_and_constant_viscosity(lat, shape, wall, force):
    N = shape[0] * shape[1]
    g = {"kind": W.G_SINE, "g0": (0.03, -0.02, 0.0), "wave_axis": 0}
    if force == "field":
        g = {"kind": W.G_FIELD, "field": 0.05 * (W.uniform(9, 30, 2 * N).reshape(2, N) - 0.5)}
    w = workload(lat, shape, tau=0.7, g=g, bc=(0, wall, 0))
    w["T_lo"], w["T_hi"] = (1.0, 1.15, 1.0), (1.0, 0.9, 1.0)
    w["rho"], w["u"], w["T"] = smooth_state(lat, shape, 12, amp_u=0.3, amp_T=0.2, amp_rho=0.2)
    if force == "mu":
        w["mu"] = 0.2
    sim, ref = lbm.Sim(w, graph_steps=2).init(), oracle_sim(w)
    sim.step(3)
    ref.step(3)
    far = np.abs(sim.populations() - ref.pulled()[perm_to_oracle(lat)])
    assert far.max() < TOL[0]


@pytest.mark.parametrize("arith", [0, 1], ids=["double", "pair"])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1e300, 1e37])
def test_what_is_not_a_state_stays_visible(bad, arith):
    w = workload(0, (40, 9, 1))
    w["fp64_arith"] = arith
    sim = lbm.Sim(w).init()
    f = sim.get_state()
    f[3, 100] = bad
    sim.set_state(f)
    sim.step(2)
    assert sim.conserved(raise_unstable=False)[0] == lbm.LBM_EUNSTABLE
