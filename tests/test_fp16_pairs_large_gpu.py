"""The FP16 step with two sites per thread, on grids that take it (65,536 sites and more on
D2Q37, 32,768 on D3Q39): the same bits as one site per thread, which is how a batch steps.

Row widths around the tiles of 64 sites, rows that share their warps between one, two and three
blocks, more and fewer rows than the wall rules touch, and one row more than a launch has room
to visit twice is in test_launch_extent_gpu."""
import numpy as np
import pytest

import paper_2302_04741_gb300 as lbm
from paper_2302_04741_gb300 import workloads as W
from helpers import workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRIDS = [(0, (64, 1024, 1)), (0, (254, 260, 1)), (0, (320, 206, 1)), (0, (2050, 32, 1)), (0, (10924, 6, 1)),
         (1, (64, 33, 16)), (1, (126, 24, 11)), (1, (320, 18, 6))]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2302_04741_gb300 import build
    build.build()


@pytest.mark.parametrize("wall", [0, 1, 2], ids=["periodic", "bounce", "thermal"])
@pytest.mark.parametrize("order,force", [(0, "uniform"), (1, "sine"), (2, "field"), (2, "mu")])
@pytest.mark.parametrize("lat,shape", GRIDS, ids=["x".join(map(str, s)) for _, s in GRIDS])
def test_same_bits_as_one_site_per_thread(lat, shape, order, force, wall):
    D, N = W.dims(lat), shape[0] * shape[1] * shape[2]
    g = {"kind": W.G_UNIFORM, "g0": (1e-3, -2e-3, 1e-3 if D == 3 else 0.0)}
    if force == "sine":  # differs between the two sites of a thread
        g = {"kind": W.G_SINE, "g0": (1e-3, 2e-3, -1e-3), "wave_axis": 0}
    if force == "field":
        g = {"kind": W.G_FIELD, "field": 2e-3 * (W.uniform(9, 30, D * N).reshape(D, N) - 0.5)}
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
