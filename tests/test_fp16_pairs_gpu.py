"""The FP16 step with two sites per thread: the same bits as one site per thread.

The batch kernel steps one site per thread (its grids are stepped by the shared
device code), so a context stepped alone and its twin in a batch must agree
exactly.  Grids: row widths around the tiles of 64 sites and the blocks of 256,
more and fewer rows than the wall rules touch, forces that differ between the
two sites of a thread, constant viscosity.
"""
import numpy as np
import pytest

import paper_2302_04741_gb300 as lbm
from paper_2302_04741_gb300 import workloads as W
from helpers import workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2302_04741_gb300 import build
    build.build()


SINE_X = {"kind": W.G_SINE, "g0": (1e-3, 2e-3, -1e-3), "wave_axis": 0}


def field_g(lat, shape):
    D, N = W.dims(lat), shape[0] * shape[1] * shape[2]
    return {"kind": W.G_FIELD, "field": 2e-3 * (W.uniform(9, 30, D * N).reshape(D, N) - 0.5)}


GRIDS = [(0, (64, 256, 1)), (0, (254, 66, 1)), (0, (256, 64, 1)), (0, (258, 64, 1)), (0, (514, 40, 1)), (0, (2050, 8, 1)),
         (1, (64, 17, 16)), (1, (126, 12, 11)), (1, (256, 7, 10)), (1, (186, 15, 6))]


@pytest.mark.parametrize("wall", [0, 1, 2], ids=["periodic", "bounce", "thermal"])
@pytest.mark.parametrize("order,force", [(0, "uniform"), (1, "sine"), (2, "uniform"), (2, "sine"), (2, "field"), (2, "mu")])
@pytest.mark.parametrize("lat,shape", GRIDS, ids=["x".join(map(str, s)) for _, s in GRIDS])
def test_same_bits_as_one_site_per_thread(lat, shape, order, force, wall):
    D = W.dims(lat)
    g = SINE_X if force == "sine" else field_g(lat, shape) if force == "field" else {"kind": W.G_UNIFORM, "g0": (1e-3, -2e-3, 1e-3 if D == 3 else 0.0)}
    bc, T_lo, T_hi = [0, 0, 0], [1.0] * 3, [1.0] * 3
    bc[D - 1], T_lo[D - 1], T_hi[D - 1] = wall, 1.1, 0.95
    w = workload(lat, shape, tau=0.6, g=g, precision=lbm.LBM_FP16_SCALED, force_order=order, bc=tuple(bc),
                 amp_u=0.2, amp_T=0.1, amp_rho=0.1)
    w["T_lo"], w["T_hi"] = tuple(T_lo), tuple(T_hi)
    if force == "mu":
        w["mu"] = 0.2
    stream = torch.cuda.Stream()
    alone, member = lbm.Sim(w, stream=stream.cuda_stream).init(), lbm.Sim(w, stream=stream.cuda_stream).init()
    b = lbm.lbm_batch_create(lat, lbm.LBM_FP16_SCALED, order, stream.cuda_stream, 1)
    try:
        lbm.lbm_batch_add(b, member.ctx)
        alone.step(3)
        lbm.lbm_batch_step(b, 3)
        assert np.array_equal(alone.get_state(), member.get_state())
    finally:
        lbm.lbm_batch_destroy(b)
