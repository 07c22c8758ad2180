"""The eight-lane FP64 step at the widest rows it takes, and the two-lane step just past them,
against the oracle (states and tolerance of test_fp64_collision_gpu)."""
import numpy as np
import pytest

import paper_2302_04741_gb300 as lbm
from helpers import oracle_sim, perm_to_oracle, smooth_state, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2302_04741_gb300 import build
    build.build()


@pytest.mark.parametrize("wall", [0, 1, 2], ids=["periodic", "bounce", "thermal"])
@pytest.mark.parametrize("shape", [(11, 9, 1), (12, 7, 1), (12, 50, 1), (13, 46, 1)], ids=["11x9", "12x7", "12x50", "13x46"])
def test_narrow_rows(shape, wall):
    g = {"kind": lbm.LBM_G_UNIFORM, "g0": (0.03, -0.05, 0.0)}
    w = workload(0, shape, tau=0.7, g=g, bc=(0, wall, 0))
    w["T_lo"], w["T_hi"] = (1.0, 1.15, 1.0), (1.0, 0.9, 1.0)
    w["rho"], w["u"], w["T"] = smooth_state(0, shape, 11, amp_u=0.3, amp_T=0.2, amp_rho=0.2)
    sim, ref = lbm.Sim(w).init(), oracle_sim(w)
    sim.step(3)
    ref.step(3)
    assert np.abs(sim.populations() - ref.pulled()[perm_to_oracle(0)]).max() < 5e-15
