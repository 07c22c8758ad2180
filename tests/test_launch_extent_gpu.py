"""Grids as tall as a launch can be (65,535 blocks along y): the step adds no rows to a
launch that has no room for them."""
import os

import numpy as np
import pytest

import oracle
import paper_2302_04741_gb300 as lbm
from paper_2302_04741_gb300 import workloads as W
from helpers import oracle_sim, perm_to_oracle, workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2302_04741_gb300 import build
    build.build()
    oracle.set_threads(os.cpu_count() or 1)


# 65,529 rows leave room for the six rows that are visited twice, 65,530 do not
@pytest.mark.parametrize("ny", [65529, 65530, 65535])
def test_fp16_rows_at_walls(ny):
    """The same bits as in a batch, whose kernel has one block index."""
    w = workload(0, (34, ny, 1), precision=lbm.LBM_FP16_SCALED, bc=(0, 2, 0), T_lo=(1.0, 1.1, 1.0), T_hi=(1.0, 0.95, 1.0))
    stream = torch.cuda.Stream()
    alone, member = lbm.Sim(w, stream=stream.cuda_stream).init(), lbm.Sim(w, stream=stream.cuda_stream).init()
    b = lbm.lbm_batch_create(0, lbm.LBM_FP16_SCALED, 2, stream.cuda_stream, 1)
    try:
        lbm.lbm_batch_add(b, member.ctx)
        alone.step(2)
        lbm.lbm_batch_step(b, 2)
        got, want = (torch.empty(37, 34 * ny, dtype=torch.float64, device="cuda") for _ in range(2))
        for sim, out in ((alone, got), (member, want)):
            lbm.lbm_get_state(sim.ctx, out)
        torch.cuda.synchronize()
        assert torch.equal(got, want)
    finally:
        lbm.lbm_batch_destroy(b)


@pytest.mark.parametrize("lat,shape", [(0, (32, 40000, 1)), (1, (8, 5, 40000))], ids=["32x40000", "8x5x40000"])
def test_sites_next_to_solids(lat, shape):
    """As many sites next to solid ones as would take the launch past its last row.  Tolerance
    per population after two steps: some 40 rounded operations on terms below 0.3 a step,
    40 x 2 x 0.3 x 2^-53 = 2.7e-15."""
    N = shape[0] * shape[1] * shape[2]
    w = workload(lat, shape)
    w["solid"] = (W.uniform(3, 8, N) < 0.3).astype(np.uint8)
    w["T_wall"] = 1.0 + 0.1 * (W.uniform(5, 9, N) - 0.5)
    sim, ref = lbm.Sim(w, block_x=32).init(), oracle_sim(w)
    sim.step(2)
    ref.step(2)
    off = np.abs(sim.populations() - ref.pulled()[perm_to_oracle(lat)])[:, w["solid"] == 0]
    assert off.max() < 2.7e-15
