"""An FP16 grid has a scale for finite fields only: one site that is not is refused."""
import numpy as np
import pytest

import paper_2302_04741_gb300 as lbm
from helpers import workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2302_04741_gb300 import build
    build.build()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("field", ["rho", "u", "T"])
@pytest.mark.parametrize("lat,shape", [(0, (67, 11, 1)), (1, (9, 7, 5))])
def test_refused(lat, shape, field, bad):
    w = workload(lat, shape, precision=lbm.LBM_FP16_SCALED)
    good = np.array(w[field])
    w[field] = np.array(good)
    w[field].reshape(-1)[-3] = bad
    sim = lbm.Sim(w)
    with pytest.raises(lbm.LbmError) as e:
        sim.init()
    assert e.value.status == lbm.LBM_EINVAL
    sim.init(**{field: good})
    sim.step(1)
