"""lbm_set_solid when an allocation fails: the context stays one that steps every fluid site.

The library's objects run on a fake CUDA runtime (fake_cudart.c), which records the kernels
that are launched and makes the n-th cudaMalloc fail."""
import ctypes
import glob
import os
import re
import subprocess

import numpy as np
import pytest

import paper_2302_04741_gb300 as lbm
from paper_2302_04741_gb300 import build as lbm_build

HERE = os.path.dirname(os.path.abspath(__file__))
SHAPE = (256, 200, 1)  # large enough for a list of wall sites
N = SHAPE[0] * SHAPE[1]
IN_PLACE, LISTED = 1, 2  # the step's template argument


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    lbm_build.build()
    so = str(tmp_path_factory.mktemp("fake") / "liblbm_fake.so")
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-o", so, os.path.join(HERE, "fake_cudart.c"),
                           *sorted(glob.glob(os.path.join(lbm_build.BUILD, "lbm_*.o"))), "-lstdc++", "-lm"])
    return so


@pytest.fixture
def fake(library, monkeypatch):
    monkeypatch.setattr(lbm, "LIB_PATH", library)
    monkeypatch.setattr(lbm, "_lib", None)
    L = lbm.lib()
    L.fake_launch_name.restype = ctypes.c_char_p
    L.fake_fail_malloc(0)
    return L


def step_launch(L, ctx):
    """(SOLID argument, rows) of a step's launch."""
    lbm.lbm_init(ctx, np.ones(N), np.zeros((2, N)), np.ones(N))
    first = L.fake_launches()
    lbm.lbm_step(ctx, 1)
    name = L.fake_launch_name(first).decode()
    return int(re.search(r"k_stepINS_5D2Q37ELi0ELi2ELi(\d)E", name).group(1)), L.fake_launch_grid(first, 1)


SOLID = np.arange(N) % 100 == 0


def create():
    return lbm.lbm_create(lbm.LBM_D2Q37, *SHAPE, 0.8)


def test_the_list_is_used(fake):
    ctx = create()
    lbm.lbm_set_solid(ctx, SOLID, np.ones(N))
    kind, rows = step_launch(fake, ctx)
    assert kind == LISTED and rows > SHAPE[1]
    lbm.lbm_destroy(ctx)


@pytest.mark.parametrize("calls", [1, 2])
def test_no_memory_for_the_list(fake, calls):
    ctx = create()
    for _ in range(calls - 1):
        lbm.lbm_set_solid(ctx, SOLID, np.ones(N))
    fake.fake_fail_malloc(5 if calls == 1 else 1)  # after the four tables
    lbm.lbm_set_solid(ctx, SOLID, np.ones(N))
    assert step_launch(fake, ctx) == (IN_PLACE, SHAPE[1])
    lbm.lbm_destroy(ctx)


@pytest.mark.parametrize("nth", [1, 2, 3, 4])
def test_no_memory_for_the_tables(fake, nth):
    ctx = create()
    before = lbm.lbm_device_bytes(ctx)
    fake.fake_fail_malloc(nth)
    with pytest.raises(lbm.LbmError) as e:
        lbm.lbm_set_solid(ctx, SOLID, np.ones(N))
    assert e.value.status == lbm.LBM_ENOMEM and lbm.lbm_device_bytes(ctx) == before
    lbm.lbm_set_solid(ctx, SOLID, np.ones(N))  # memory has come back
    assert step_launch(fake, ctx)[0] == LISTED
    lbm.lbm_destroy(ctx)
