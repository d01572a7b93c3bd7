"""The middle of the ranges of lbmp_step's default kernels, bit for bit against the
single-step ones: FP16 lattices between the tiles' range and the strips of two
pairs a lane (one pair a lane: narrow, odd, static and dynamic Kn, both roundings),
and the largest FP32 lattices that run on tiles.  The launches are counted, so that
a lattice that goes another way fails here."""
import numpy as np
import pytest

from paper_1411_7051_gb300 import media
from helpers import Case, gpu_sim

pytestmark = pytest.mark.gpu

REST = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
AUTO, STAGED, DIRECT = 0, 1, 2


def _run(case, storage, kernel, rounding, steps):
    f0 = media.random_populations(case.nx, case.ny, seed=3, base=REST, amp=2e-3)
    with gpu_sim(case, storage, kernel=kernel, fp16_rounding=rounding, seed=5) as s:
        s.set_populations(f0)
        before = s.info().launches
        for n in steps:
            s.step(n)
        launches = s.info().launches - before
        return s.populations(), launches


def _case(nx, ny, walls, pressure, forch, beta):
    med = media.random_medium(nx, ny, seed=nx + ny, p_open=0.1, p_solid=0.1,
                              log10_k_range=(-3, 0), kn_range=(0.0, 5.0))
    return Case(nx, ny, tau=0.7, G=(1e-5, 3e-6), walls=walls, pressure=pressure, rho_in=1.001,
                rho_out=0.999, forchheimer=forch, medium=med, kn_beta=beta)


@pytest.mark.parametrize("walls,pressure", [(False, False), (True, False), (False, True),
                                            (True, True)])
@pytest.mark.parametrize("nx,ny", [(64, 1200), (65, 1201), (125, 601), (127, 900), (301, 400),
                                   (500, 401), (1301, 60), (8191, 12), (999, 1000)])
def test_fp16_one_pair_a_lane(nx, ny, walls, pressure):
    for forch, beta, rounding in ((1, 0.0, 0), (0, 0.0, 1), (1, 100.0, 0), (0, 100.0, 1)):
        case = _case(nx, ny, walls, pressure, forch, beta)
        fa, la = _run(case, 1, AUTO, rounding, (2, 1, 5))
        fb, lb = _run(case, 1, STAGED, rounding, (2, 1, 5))
        assert bool((fa == fb).all()), f"{int((fa != fb).sum())} populations differ"
        # pairs 1 + 0 + 2, single steps 0 + 1 + 1, and with stochastic rounding a
        # counter bump for each of the four groups of them
        assert la == 5 + (4 if rounding == 0 else 0) and lb > la


@pytest.mark.parametrize("walls,pressure", [(False, False), (True, True)])
@pytest.mark.parametrize("nx,ny", [(410, 413), (131, 1290), (1695, 100), (41, 4000)])
def test_fp32_largest_tiles(nx, ny, walls, pressure):
    steps = (16, 19, 40)
    for forch, beta in ((1, 0.0), (0, 100.0)):
        case = _case(nx, ny, walls, pressure, forch, beta)
        fa, la = _run(case, 0, AUTO, 0, steps)
        fb, lb = _run(case, 0, DIRECT, 0, steps)
        assert bool((fa == fb).all()), f"{int((fa != fb).sum())} populations differ"
        # at least four steps a launch (a remainder of two may take two launches)
        assert lb == sum(steps) and la <= sum(n // 4 + 2 for n in steps)
