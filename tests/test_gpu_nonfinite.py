"""Read-outs of a lattice with a non-finite node: the sums and the histogram
report it (ENAN) without touching their outputs, the fields show the node, and
the same lattice reads out as usual once its populations are finite again."""
import ctypes

import numpy as np
import pytest

from paper_1411_7051_gb300 import lbmp, media
from helpers import Case, gpu_sim

pytestmark = pytest.mark.gpu

REST = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("storage,beta", [(0, 0.0), (0, 100.0), (1, 0.0), (1, 100.0)])
@pytest.mark.parametrize("nx,ny", [(7, 6), (300, 41)])
def test_nonfinite_node_is_reported(nx, ny, storage, beta, value):
    med = media.random_medium(nx, ny, seed=1, p_open=0.1, p_solid=0.0, log10_k_range=(-3, 0),
                              kn_range=(0.0, 5.0))
    case = Case(nx, ny, tau=0.7, G=(1e-5, 3e-6), walls=True, pressure=True, rho_in=1.001,
                rho_out=0.999, forchheimer=1, medium=med, kn_beta=beta)
    good = media.random_populations(nx, ny, seed=3, base=REST, amp=2e-3)
    bad = good.copy()
    bad[5, 2, 3] = value
    with gpu_sim(case, storage, seed=5) as s:
        s.set_populations(bad)
        for read in (s.permeability, s.mass, s.residual, lambda: s.velocity_histogram(10)):
            with pytest.raises(lbmp.LbmpError) as e:
                read()
            assert e.value.status == lbmp.ENAN
        counts = (ctypes.c_int64 * 10)(*[-7] * 10)
        umax = ctypes.c_double(-7.0)
        assert lbmp.load().lbmp_velocity_histogram(s._h, 10, ctypes.byref(umax),
                                                   counts) == lbmp.ENAN
        assert list(counts) == [-7] * 10 and umax.value == -7.0
        fields = [f.cpu().numpy() for f in s.macroscopic()]
        assert not all(np.isfinite(f[2, 3]) for f in fields)
        for f in fields:
            f[2, 3] = 0.0
            assert np.isfinite(f).all()
        s.set_populations(good)
        counts, umax = s.velocity_histogram(10)
        assert int(np.asarray(counts).sum()) == nx * (ny - 2) and umax > 0
        s.residual()
        assert np.isfinite(s.residual()) and np.isfinite(s.permeability()[0])
