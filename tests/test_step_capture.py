"""lbmp_step on a stream that is being captured is refused, whatever the number
of steps, before the lattice's own state moves on: its graphs cannot be recorded
into another one, and a replay could not alternate the two buffers.  Host logic,
against a runtime without a GPU that refuses a graph launch there as CUDA does."""
import ctypes

import pytest

import fake_device as fake
from paper_1411_7051_gb300 import lbmp

STREAM = 0x77


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    return fake.load(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("nx,ny,kw", [(64, 33, {}), (64, 33, dict(storage=1)), (410, 200, {}),
                                      (200, 200, dict(kn_beta=100.0)), (600, 500, dict(storage=1)),
                                      (512, 512, {}), (1024, 1024, {})])
def test_capture_is_refused(L, nx, ny, kw, warm):
    for n in (1, 2, 3, 5, 7, 11, 15, 33, 64):
        st, h = fake.create(L, fake.params(nx, ny, stream=STREAM, **kw))
        assert st == lbmp.OK
        if warm:
            assert L.lbmp_step(h, n) == L.lbmp_step(h, n) == lbmp.OK
        before, after = lbmp.Info(), lbmp.Info()
        L.lbmp_get_info(h, ctypes.byref(before))
        L.fake_capture(STREAM, 1)
        st = L.lbmp_step(h, n)
        L.fake_capture(STREAM, 0)
        assert st == lbmp.ECUDA, n
        L.lbmp_get_info(h, ctypes.byref(after))
        assert (after.steps, after.launches) == (before.steps, before.launches)
        assert L.lbmp_step(h, n) == lbmp.OK
        L.lbmp_destroy(h)


@pytest.mark.parametrize("nx,ny,direct", [(64, 33, 1), (40, 4000, 1), (128, 64, 2), (410, 200, 2),
                                          (3000, 56, 2)])
def test_few_steps_of_a_small_fp32_lattice_run_the_direct_kernel(L, nx, ny, direct):
    """One step, and two on lattices that fill the direct kernel's blocks, cost
    less without the halo of a tile."""
    for n in (1, 2, 3):
        st, h = fake.create(L, fake.params(nx, ny))
        tile, step = (L.fake_launches(k) for k in (b"16tile_step_kernel", b"11step_kernel"))
        assert L.lbmp_step(h, n) == lbmp.OK
        assert L.fake_launches(b"16tile_step_kernel") == tile + (n > direct)
        assert L.fake_launches(b"11step_kernel") == step + (n if n <= direct else 0)
        L.lbmp_destroy(h)
