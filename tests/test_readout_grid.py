"""Blocks of a read-out: whole waves of the chip or at least half a wave more,
never the few blocks beyond the first wave that take as long as a second one.
Host logic, against a runtime without a GPU."""
import pytest

import fake_device as fake
from paper_1411_7051_gb300 import lbmp

WAVE = 4 * 152   # four blocks on each multiprocessor


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    return fake.load(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("nx,ny,waves", [(64, 33, 0), (1, 65535, 1), (40, 65535, 1), (257, 12000, 1),
                                         (1500, 2400, 1), (1600, 2400, 1.5), (257, 30000, 3),
                                         (4096, 4096, 4), (1000000, 4, 6)])
def test_no_nearly_empty_second_wave(L, nx, ny, waves):
    p = fake.params(nx, ny, bc_x=lbmp.BCX_PERIODIC, rho_in=1.0, rho_out=1.0, G=(1e-6, 0.0))
    st, h = fake.create(L, p)
    assert st == lbmp.OK
    assert L.lbmp_macroscopic(h, None, None, None, lbmp.DEVICE) == lbmp.OK
    blocks = L.fake_blocks(b"13fields_kernel")
    assert blocks <= WAVE or blocks >= 1.4 * WAVE
    assert int(blocks / WAVE + 0.1) == int(waves)   # (rows are dealt out to whole columns)
    L.lbmp_destroy(h)
