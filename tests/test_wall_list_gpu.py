"""FP64 grids large enough for a list of the fluid sites next to solid ones (28,672 sites and
more): which of them keep it, and their steps against the oracle.

The list is kept where it saves work: with L sites in it, W warps (32 sites of a row) that
have one and M that have one and another fluid site too, where M + L / 16 <= 2 W.

Tolerance per population after three steps: some 40 rounded operations on terms below 0.3 a
step, 40 x 3 x 0.3 x 2^-53 = 4e-15.
"""
import os

import numpy as np
import pytest

import oracle
import paper_2302_04741_gb300 as lbm
from paper_2302_04741_gb300 import workloads as W
from helpers import oracle_sim, perm_to_oracle, workload

pytestmark = pytest.mark.gpu

KEPT = {"corner": True, "slab": True, "few": True, "some": False, "many": True}


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
    return W.uniform(3, 8, nx * ny * nz) < {"few": 0.004, "some": 0.06, "many": 0.3}[kind]


def listed_sites(lat, shape, solid):
    """L, and whether the list is kept."""
    nx, ny, nz = shape
    s = solid.reshape(nz, ny, nx)
    near = np.zeros_like(s)
    for e in lbm.lbm_lattice_info(lat)[3]:
        near |= np.roll(s, (e[2], e[1], e[0]), (0, 1, 2))
    wall = near & ~s
    warps = lambda v: np.pad(v, ((0, 0), (0, 0), (0, -nx % 32))).reshape(nz, ny, -1, 32).any(3)  # noqa: E731
    has, other = warps(wall), warps(~near & ~s)
    return int(wall.sum()), (has & other).sum() + wall.sum() / 16.0 <= 2 * has.sum()


@pytest.mark.parametrize("sigma", [False, True])
@pytest.mark.parametrize("kind", list(KEPT))
@pytest.mark.parametrize("lat,shape", [(0, (233, 131, 1)), (1, (63, 22, 21))], ids=["233x131", "63x22x21"])
def test_steps(lat, shape, kind, sigma):
    N = shape[0] * shape[1] * shape[2]
    w = workload(lat, shape)
    w["mu"], w["include_sigma"] = 0.25, sigma
    solid = mask(kind, shape)
    w["solid"], w["T_wall"] = solid.astype(np.uint8), 1.0 + 0.1 * (W.uniform(5, 9, N) - 0.5)
    n, kept = listed_sites(lat, shape, solid)
    assert kept == KEPT[kind]
    sim = lbm.Sim(w)
    before = lbm.lbm_device_bytes(sim.ctx)
    lbm.lbm_set_solid(sim.ctx, w["solid"], w["T_wall"])
    # tables of 14 bytes a site, and the list
    assert lbm.lbm_device_bytes(sim.ctx) - before == 14 * N + (4 * n if kept else 0)
    sim.init()
    ref = oracle_sim(w)
    sim.step(3)
    ref.step(3)
    off = np.abs(sim.populations() - ref.pulled()[perm_to_oracle(lat)])[:, ~solid]
    assert off.max() < 5e-15
