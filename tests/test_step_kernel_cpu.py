"""Which kernel a step launches, by grid and storage (fake CUDA runtime, see test_set_solid_cpu)."""
import numpy as np
import pytest

import paper_2302_04741_gb300 as lbm
from test_set_solid_cpu import fake, library  # noqa: F401 (fixtures)


def kernel(L, lat, shape, **options):
    o = lbm.lbm_default_options()
    for k, v in options.items():
        setattr(o, k, v)
    ctx = lbm.lbm_create(lat, *shape, 0.8, None, o)
    N = shape[0] * shape[1] * shape[2]
    lbm.lbm_init(ctx, np.ones(N), np.zeros((2 + lat, N)), np.ones(N))
    first = L.fake_launches()
    lbm.lbm_step(ctx, 1)
    lbm.lbm_destroy(ctx)
    return L.fake_launch_name(first).decode()


# 8 lanes a site multiply the FP64 work by four: for narrow rows only
@pytest.mark.parametrize("shape,name", [((3, 150, 1), "k_step_splitILi2ELi8E"), ((12, 50, 1), "k_step_splitILi2ELi8E"),
                                        ((13, 46, 1), "k_step_symILi2E"), ((32, 19, 1), "k_step_symILi2E"),
                                        ((12, 51, 1), "k_step_symILi2E"), ((64, 152, 1), "k_step_symILi2E"),
                                        ((64, 153, 1), "k_stepINS_5D2Q37ELi0E")])
def test_lanes_of_the_fp64_step(fake, shape, name):  # noqa: F811
    assert name in kernel(fake, lbm.LBM_D2Q37, shape)


# two sites a thread: even rows, grids large enough that a thread's latency does not count
@pytest.mark.parametrize("lat,shape,two", [(0, (512, 128, 1), True), (0, (510, 128, 1), False), (0, (513, 128, 1), False),
                                           (0, (256, 192, 1), False), (1, (64, 32, 16), True), (1, (64, 31, 16), False)])
def test_sites_per_thread_of_the_fp16_step(fake, lat, shape, two):  # noqa: F811
    name = kernel(fake, lat, shape, precision=lbm.LBM_FP16_SCALED)
    assert ("k_step_half2" in name) == two
