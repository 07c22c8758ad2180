"""Batches with more tiles than CTAs: a CTA takes a run of consecutive tiles, over
the ends of grids; when members leave, the launch shrinks.  Each grid must come out
bit-identical to the same grid stepped alone."""
import numpy as np
import pytest

import paper_2302_04741_gb300 as lbm
from paper_2302_04741_gb300 import workloads as W
from helpers import workload

pytestmark = pytest.mark.gpu

# about 2.5 million sites: 16 waves of resident blocks hold up to 2
BIG = {0: [((1501, 1003, 1), (0, 2, 0)), ((2050, 501, 1), (0, 0, 0))],
       1: [((131, 97, 101), (0, 0, 2)), ((128, 128, 77), (0, 0, 0))]}
SMALL = {0: [((36, 40, 1), (0, 0, 0)), ((67, 9, 1), (0, 1, 0)), ((8, 8, 1), (0, 0, 0))],
         1: [((16, 9, 8), (0, 0, 0)), ((9, 8, 16), (0, 0, 2)), ((7, 7, 7), (0, 0, 0))]}


@pytest.mark.parametrize("lat,precision,cfg", [
    (0, 1, (64, 1, 4)), (0, 1, (256, 1, 0)), (0, 2, (128, 1, 4)), (1, 1, (128, 1, 0)), (1, 2, (64, 1, 0))])
def test_runs_bitwise_equal_single(lat, precision, cfg):
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    big, small = BIG[lat], SMALL[lat]
    specs = [small[0], big[0], small[1], small[2], big[1], small[0]]
    ws = [workload(lat, shape, tau=0.55 + 0.1 * k, seed=40 + k, precision=precision, bc=bc,
                   T_lo=(1.0, 1.06, 1.06), T_hi=(1.0, 0.95, 0.95),
                   g={"kind": W.G_UNIFORM, "g0": (1e-5 * (k + 1), -2e-5, 1e-5)})
          for k, (shape, bc) in enumerate(specs)]
    members = [lbm.Sim(w, stream=stream.cuda_stream).init() for w in ws]
    alone = [lbm.Sim(w).init() for w in ws]
    b = lbm.lbm_batch_create(lat, precision, 2, stream.cuda_stream, 16)
    try:
        for m in members:
            lbm.lbm_batch_add(b, m.ctx)
        lbm.lbm_batch_set_config(b, *cfg)
        lbm.lbm_batch_step(b, 9)
        for a in alone:
            a.step(9)
        for m, a in zip(members, alone):
            np.testing.assert_array_equal(m.get_state(), a.get_state())
        left = [0, 2, 3, 5]
        for k in (1, 4):
            lbm.lbm_batch_remove(b, members[k].ctx)
        lbm.lbm_batch_step(b, 5)  # a launch of fewer blocks
        if precision == 1:        # and through the other kernel and back
            lbm.lbm_batch_set_staging(b, 1)
            lbm.lbm_batch_step(b, 5)
            lbm.lbm_batch_set_staging(b, 0)
        lbm.lbm_batch_add(b, members[1].ctx)
        lbm.lbm_batch_step(b, 5)
        for k in left:
            alone[k].step(15 if precision == 1 else 10)
        alone[1].step(5)
        for k in left + [1]:
            np.testing.assert_array_equal(members[k].get_state(), alone[k].get_state())
    finally:
        lbm.lbm_batch_destroy(b)
