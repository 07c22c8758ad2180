"""Grids with solid sites: the fluid sites next to a solid one are stepped from a
list, in blocks of their own, the others with the plain pull.  Masks of scattered
sites (nearly every fluid site in the list, and few), a slab, and one solid
corner across the periodic edges, against the oracle.

Tolerance per population after three steps: some 40 rounded operations on terms
below 0.3 a step, 40 x 3 x 0.3 x 2^-53 = 4e-15 in double; in float, with 2^-24,
2.1e-6.
"""
import os

import numpy as np
import pytest

import oracle
import paper_2302_04741_gb300 as lbm
from paper_2302_04741_gb300 import workloads as W
from helpers import oracle_sim, perm_to_oracle, workload

pytestmark = pytest.mark.gpu

TOL = {lbm.LBM_FP64: 5e-15, lbm.LBM_FP32_SHIFTED: 2.2e-6}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2302_04741_gb300 import build
    build.build()
    oracle.set_threads(os.cpu_count() or 1)


def mask(kind, shape):
    nx, ny, nz = shape
    zz, yy, xx = np.indices((nz, ny, nx)).reshape(3, nx * ny * nz)
    if kind == "corner":
        return (xx < 2) & (yy < 2) & (zz < 2)
    if kind == "slab":
        return (yy >= 3) & (yy < 7)
    return W.uniform(3, 8, nx * ny * nz) < (0.004 if kind == "few" else 0.3)


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["few", "many", "slab", "corner"])
@pytest.mark.parametrize("lat,shape", [(0, (67, 41, 1)), (0, (130, 20, 1)), (1, (35, 11, 9))], ids=["67x41", "130x20", "35x11x9"])
def test_steps_and_sums(lat, shape, kind, precision):
    N = shape[0] * shape[1] * shape[2]
    w = workload(lat, shape, precision=precision, force_order=2)
    w["mu"] = 0.25
    w["solid"] = mask(kind, shape).astype(np.uint8)
    w["T_wall"] = 1.0 + 0.1 * (W.uniform(5, 9, N) - 0.5)
    sim, ref = lbm.Sim(w).init(), oracle_sim(w)
    sim.step(3)
    ref.step(3)
    fluid = w["solid"] == 0
    far = np.abs(sim.populations() - ref.pulled()[perm_to_oracle(lat)])[:, fluid]
    assert far.max() < TOL[precision]
    got, want = sim.moments(), ref.moments()
    for a, b in zip(got[:3], want[:3]):
        assert np.abs(np.asarray(a)[..., fluid] - np.asarray(b)[..., fluid]).max() < 300 * TOL[precision]
    _, mass, _, _ = sim.conserved()
    assert abs(mass - want[0][fluid].sum()) < 10 * TOL[precision] * N
