"""The scale that lbm_init chooses for FP16 storage: s = 2^k with the largest
|f~_i - w_i| / w_i of the initial state times s in [2^12, 2^13).

The largest deviation is placed in one direction, at the last site of a grid
that fills no block, and elsewhere; the state comes from the float-precision
init, which leaves a deviation of 0.01 its leading 5 digits, so amplitudes stay
1e-3 away from the powers of two between which k changes.
"""
import numpy as np
import pytest

import paper_2302_04741_gb300 as lbm
from paper_2302_04741_gb300 import workloads as W
from helpers import oracle_sim, perm_to_oracle, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2302_04741_gb300 import build
    build.build()


@pytest.mark.parametrize("lat,shape", [(0, (3, 3, 1)), (0, (257, 5, 1)), (0, (700, 613, 1)), (1, (5, 3, 4)), (1, (65, 66, 67))])
@pytest.mark.parametrize("where", ["first", "last"])
def test_scale_of_the_largest_deviation(lat, shape, where):
    D, N = W.dims(lat), shape[0] * shape[1] * shape[2]
    w = workload(lat, shape, precision=lbm.LBM_FP16_SCALED, amp_u=0.0, amp_T=0.0, amp_rho=1e-3)
    at = 0 if where == "first" else N - 1
    w["u"] = np.zeros((D, N))
    w["u"][D - 1, at] = 0.1
    sim = lbm.Sim(w).init()
    # the largest |f~_i - w_i| / w_i, at that site, from the oracle's init (periodic: its pulled state)
    small = dict(w, shape=(3, 3, 3 if D == 3 else 1))
    n = 3 ** D
    small.update(rho=np.full(n, w["rho"][at]), u=np.repeat(w["u"][:, at:at + 1], n, 1), T=np.full(n, w["T"][at]))
    f = oracle_sim(small).pulled()[perm_to_oracle(lat)][:, 0]
    wts = lbm.lbm_lattice_info(lat)[4]
    big = float(np.max(np.abs(f - wts) / wts))
    assert abs(np.log2(big) - round(np.log2(big))) > 1e-3
    assert lbm.lbm_fp16_scale(sim.ctx) == 2.0 ** (12 - int(np.floor(np.log2(big))))

