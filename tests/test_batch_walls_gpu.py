"""Batches whose members have walls, have none, or are mixed: a batch of grids without walls
runs a kernel of its own, and changes it when a member with walls comes or goes.  The bits are
those of each grid stepped alone."""
import numpy as np
import pytest

import paper_2302_04741_gb300 as lbm
from helpers import workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# rows shorter and longer than a warp, tiles that start in a wall row and between them
GRIDS = {0: [(19, 7, 1), (130, 11, 1), (33, 40, 1)], 1: [(19, 6, 7), (40, 5, 13), (66, 4, 6)]}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2302_04741_gb300 import build
    build.build()


@pytest.mark.parametrize("order", [0, 2])
@pytest.mark.parametrize("wall", [1, 2], ids=["bounce", "thermal"])
@pytest.mark.parametrize("precision", [1, 2], ids=["fp32", "fp16"])
@pytest.mark.parametrize("lat", [0, 1], ids=["D2Q37", "D3Q39"])
def test_members_come_and_go(lat, precision, wall, order):
    stream = torch.cuda.Stream()

    def pair(k, shape, with_wall):
        bc, T_lo, T_hi = [0, 0, 0], [1.0] * 3, [1.0] * 3
        if with_wall:
            bc[1 + lat], T_lo[1 + lat], T_hi[1 + lat] = wall, 1.1, 0.95
        w = workload(lat, shape, tau=0.6 + 0.1 * k, seed=3 + k, precision=precision, force_order=order, bc=tuple(bc),
                     T_lo=tuple(T_lo), T_hi=tuple(T_hi), amp_u=0.1, amp_T=0.05)
        return tuple(lbm.Sim(w, stream=stream.cuda_stream).init() for _ in range(2))

    plain = [pair(k, s, False) for k, s in enumerate(GRIDS[lat])]
    walled = [pair(3 + k, s, True) for k, s in enumerate(GRIDS[lat])]
    b = lbm.lbm_batch_create(lat, precision, order, stream.cuda_stream, 6)
    lbm.lbm_batch_set_config(b, 128, 1, 2)

    def step(members):
        lbm.lbm_batch_step(b, 5)
        for alone, _ in members:
            alone.step(5)
        for alone, member in members:
            np.testing.assert_array_equal(alone.get_state(), member.get_state())

    try:
        for _, m in plain:
            lbm.lbm_batch_add(b, m.ctx)
        step(plain)
        for _, m in walled:
            lbm.lbm_batch_add(b, m.ctx)
        step(plain + walled)
        for _, m in plain:
            lbm.lbm_batch_remove(b, m.ctx)
        step(walled)
        for _, m in walled:
            lbm.lbm_batch_remove(b, m.ctx)
        for _, m in plain:
            lbm.lbm_batch_add(b, m.ctx)
        step(plain)
    finally:
        lbm.lbm_batch_destroy(b)
