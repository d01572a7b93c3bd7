"""The split of a two-step launch is planned once per lattice, not per launch:
a narrow tall lattice has thousands of candidate splits, and its calls must not
cost the host more than those of a square one with the same launches.  Host
logic, against a runtime without a GPU."""
import ctypes
import time

import numpy as np
import pytest

import fake_device as fake
from paper_1411_7051_gb300 import lbmp


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    return fake.load(tmp_path_factory.mktemp("fake"))


def _first_step(L, nx, ny):
    st, h = fake.create(L, fake.params(nx, ny))
    t = time.perf_counter()
    assert L.lbmp_step(h, 101) == lbmp.OK
    t = time.perf_counter() - t
    L.lbmp_destroy(h)
    return t


def _gradient(L, nx, ny):
    st, h = fake.create(L, fake.params(nx, ny))
    out = np.zeros(2 * nx * ny).ctypes.data
    vp = ctypes.c_void_p
    t = time.perf_counter()
    assert L.lbmp_permeability_gradient(h, 400, 0, None, vp(out), vp(out + 8 * nx * ny),
                                        lbmp.DEVICE) == lbmp.OK
    t = time.perf_counter() - t
    L.lbmp_destroy(h)
    return t


@pytest.mark.parametrize("call", [_first_step, _gradient])
def test_plan_is_not_searched_per_launch(L, call):
    narrow = min(call(L, 64, 8192) for _ in range(7))
    square = min(call(L, 512, 1024) for _ in range(7))
    assert narrow < 2.5 * square
