"""The two-step kernel (lbmp_step with the default kernel choice) against the
single-step kernels, bit for bit: FP16 storage against the staged kernel (the
same stochastic-rounding bits), FP32 against the direct one.  Sizes: strips of
64 and 128 columns with their overlaps and remainders, odd widths, the smallest
lattices taken, single-row segments and long ones."""
import numpy as np
import pytest

from paper_1411_7051_gb300 import media
from helpers import Case, gpu_sim

pytestmark = pytest.mark.gpu

FP32, FP16 = 0, 1
AUTO, STAGED, DIRECT = 0, 1, 2
REST = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


def _case(nx, ny, walls, pressure, forch, beta, p_solid=0.1):
    med = media.random_medium(nx, ny, seed=nx + ny, p_open=0.1, p_solid=p_solid,
                              log10_k_range=(-3, 0), kn_range=(0.0, 5.0))
    return Case(nx, ny, tau=0.7, G=(1e-5, 3e-6), walls=walls, pressure=pressure, rho_in=1.001,
                rho_out=0.999, forchheimer=forch, medium=med, kn_beta=beta)


def _same(case, storage, other, rounding=0):
    f0 = media.random_populations(case.nx, case.ny, seed=3, base=REST, amp=2e-3)
    out = []
    for kernel in (AUTO, other):
        s = gpu_sim(case, storage, kernel=kernel, fp16_rounding=rounding, seed=5)
        s.set_populations(f0)
        for n in (2, 1, 5):   # whole pairs, a single step, pairs and a single step
            s.step(n)
        out.append(s)
    a, b = out
    # the default choice ran steps in pairs: 4 launches of two steps or one
    # less than the 8 single ones (each call's counter bump aside)
    assert a.info().launches < b.info().launches
    fa, fb = a.populations(), b.populations()
    assert a.info().steps == b.info().steps == 8
    assert bool((fa == fb).all()), f"{int((fa != fb).sum())} populations differ"
    a.close()
    b.close()


@pytest.mark.parametrize("walls,pressure", [(False, False), (True, False), (False, True),
                                            (True, True)])
@pytest.mark.parametrize("nx,ny", [(64, 6), (65, 7), (124, 12), (125, 12), (127, 9), (128, 33),
                                   (185, 20), (301, 41), (1003, 1001), (8192, 130)])
def test_fp16_matches_staged(nx, ny, walls, pressure):
    for forch, beta, rounding in ((1, 0.0, 0), (0, 0.0, 1), (1, 100.0, 0)):
        _same(_case(nx, ny, walls, pressure, forch, beta), FP16, STAGED, rounding)


@pytest.mark.parametrize("walls,pressure", [(False, False), (True, True)])
@pytest.mark.parametrize("nx,ny,beta", [(64, 8192, 0.0), (125, 4200, 0.0), (1000, 510, 0.0),
                                        (129, 8001, 0.0), (1003, 1001, 0.0), (1003, 1001, 100.0),
                                        (16390, 64, 0.0), (16391, 64, 100.0)])
def test_fp32_matches_direct(nx, ny, beta, walls, pressure):
    for forch in (0, 1):
        _same(_case(nx, ny, walls, pressure, forch, beta), FP32, DIRECT)


def test_permeable_everywhere_and_nowhere():
    """The straight-line form of a row (every node of a warp permeable) and
    the general one (a lattice of impermeable nodes)."""
    for p_solid in (0.0, 1.0):
        case = _case(1024, 520, True, True, 1, 0.0, p_solid)
        _same(case, FP32, DIRECT)
        _same(case, FP16, STAGED)


@pytest.mark.parametrize("walls,pressure", [(False, False), (True, True)])
@pytest.mark.parametrize("storage,rounding", [(FP32, 0), (FP16, 0), (FP16, 1)])
@pytest.mark.parametrize("sizes", [[(64, 6), (131, 20), (256, 64), (300, 41), (65, 9)],
                                   [(128, 400), (1024, 513), (1003, 700)]])
def test_batch_pairs_match_single_steps(sizes, storage, rounding, walls, pressure):
    """The staged candidate advances a batch two steps per launch; steps asked
    for one by one run its single-step kernel.  Both give the same bits."""
    from paper_1411_7051_gb300 import lbmp
    cfg = lbmp.SimConfig(1, 1, tau=0.75, G=(1e-5, 2e-6), forchheimer=1, storage=storage,
                         bc_x=lbmp.BCX_PRESSURE if pressure else lbmp.BCX_PERIODIC,
                         bc_y=lbmp.BCY_WALLS if walls else lbmp.BCY_PERIODIC, rho_in=1.001,
                         rho_out=0.999, fp16_rounding=rounding, seed=11)
    out = []
    for pairs in (True, False):
        with lbmp.Batch(cfg, sizes) as b:
            b.set_shape(9)
            for i, (nx, ny) in enumerate(sizes):
                m = media.random_medium(nx, ny, seed=i, p_open=0.1, p_solid=0.05,
                                        log10_k_range=(-3, 0))
                b.set_fields(i, m.eps, m.k_i, m.kn)
            launches = b.info().launches
            for n in (37, 4):   # one graph replay of 32 steps, pairs and a single step
                if pairs:
                    b.step(n)
                else:
                    for _ in range(n):
                        b.step(1)
            b.synchronize()
            out.append(([b.populations(i) for i in range(len(sizes))], b.permeability()[0],
                        b.info().launches - launches))
    (pa, ka, la), (pb, kb, lb) = out
    assert la < lb
    for fa, fb in zip(pa, pb):
        assert bool((fa == fb).all()), f"{int((fa != fb).sum())} populations differ"
    assert np.array_equal(ka, kb)
