"""Several steps per launch on small lattices (lbmp_step with the default kernel
choice) against the single-step kernels, bit for bit: FP32 against the direct
kernel, FP16 against the staged one.  Sizes: one node, one row or column, tiles of
unequal widths, columns beyond one warp, the largest taken."""
import numpy as np
import pytest

from paper_1411_7051_gb300 import media
from helpers import Case, gpu_sim

pytestmark = pytest.mark.gpu

REST = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


@pytest.mark.parametrize("walls,pressure", [(False, False), (True, False), (False, True),
                                            (True, True)])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 5), (5, 1), (3, 3), (7, 6), (64, 33), (65, 7),
                                   (131, 37), (300, 41), (410, 170), (2000, 5), (5, 2000)])
def test_matches_single_steps(nx, ny, walls, pressure):
    if walls and ny < 3 or pressure and nx < 3:
        pytest.skip("lattice too small for this boundary kind")
    med = media.random_medium(nx, ny, seed=nx + ny, p_open=0.1, p_solid=0.1,
                              log10_k_range=(-3, 0), kn_range=(0.0, 5.0))
    f0 = media.random_populations(nx, ny, seed=3, base=REST, amp=2e-3)
    for storage, rounding, forch, beta in ((0, 0, 1, 0.0), (0, 0, 0, 100.0), (1, 0, 1, 0.0),
                                           (1, 1, 0, 100.0)):
        case = Case(nx, ny, tau=0.7, G=(1e-5, 3e-6), walls=walls, pressure=pressure, rho_in=1.001,
                    rho_out=0.999, forchheimer=forch, medium=med, kn_beta=beta)
        out = []
        for kernel in (0, 1 if storage else 2):
            s = gpu_sim(case, storage, kernel=kernel, fp16_rounding=rounding, seed=5)
            s.set_populations(f0)
            before = s.info().launches
            for n in (1, 2, 16, 19, 40):   # remainders of one and more steps, whole launches
                s.step(n)
            out.append((s.populations(), s.info().launches - before))
            assert s.info().steps == 78
            s.close()
        (fa, la), (fb, lb) = out
        assert bool((fa == fb).all()), f"{int((fa != fb).sum())} populations differ"
        if nx * ny <= 70000:
            assert 2 * la < lb   # several steps per launch
