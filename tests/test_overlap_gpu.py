"""Steps launched as programmatic dependents of the step before: on a grid of more
blocks than fit at once the first blocks of a step run beside the last ones of the
step before, and must not read what those still write."""
import numpy as np
import pytest

import paper_2302_04741_gb300 as lbm
from paper_2302_04741_gb300 import workloads as W
from helpers import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,shape,bc", [
    (0, (2050, 501, 1), (0, 0, 0)), (0, (1030, 700, 1), (0, 2, 0)), (0, (1001, 703, 1), (0, 0, 0)),
    (1, (98, 90, 100), (0, 0, 0)), (1, (91, 90, 100), (0, 0, 2))])
@pytest.mark.parametrize("force", ["uniform", "sine"])
@pytest.mark.parametrize("order", [0, 2])
@pytest.mark.parametrize("precision,opt", [(0, {}), (0, {"fp64_arith": 1}), (1, {}), (2, {})])
def test_overlapped_steps_of_many_blocks(lat, shape, bc, precision, opt, order, force):
    g = {"kind": W.G_UNIFORM, "g0": (1e-5, -2e-5, 1e-5)}
    if force == "sine":
        g = {"kind": W.G_SINE, "g0": (1e-3, 2e-3, -1e-3), "wave_axis": 1}
    w = workload(lat, shape, seed=11, precision=precision, force_order=order, bc=bc, T_lo=(1.0, 1.06, 1.06),
                 T_hi=(1.0, 0.95, 0.95), g=g)
    a = lbm.Sim(w, overlap_steps=1, **opt).init()
    b = lbm.Sim(w, overlap_steps=0, **opt).init()
    for n in (1, 2, 6):
        a.step(n)
        b.step(n)
        np.testing.assert_array_equal(a.get_state(), b.get_state())


@pytest.mark.parametrize("precision", [0, 1])
def test_overlapped_steps_with_solids(precision):
    shape = (1030, 700, 1)
    w = workload(0, shape, seed=12, precision=precision)
    w["T_wall"] = np.ones(shape[0] * shape[1])
    rng = np.random.default_rng(3)
    w["solid"] = (rng.random((shape[1], shape[0])) < 0.02).astype(np.uint8).ravel()
    a = lbm.Sim(w, overlap_steps=1).init()
    b = lbm.Sim(w, overlap_steps=0).init()
    for n in (1, 2, 6):
        a.step(n)
        b.step(n)
        np.testing.assert_array_equal(a.get_state(), b.get_state())
