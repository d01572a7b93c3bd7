"""The read-outs against each other and against numpy on the same values: FP64
fields formed with integer operations are exact, the sums agree with sums over
the fields, the histogram replays bin by bin also where its FP32 estimates do
not apply.  Sizes: one row or column, odd ones, rows that leave a lone node or a
block without work."""
import numpy as np
import pytest

from paper_1411_7051_gb300 import media
from helpers import Case, gpu_sim

pytestmark = pytest.mark.gpu

W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
SIZES = [(1, 5), (5, 1), (257, 3), (130, 613), (3000, 7), (64, 33)]


def _np(t):
    return t.detach().cpu().numpy()


def _sim(nx, ny, storage, beta=0.0, pressure=False, g=(2e-5, 4e-6), p_solid=0.1, steps=6):
    walls = ny >= 3
    med = media.random_medium(nx, ny, seed=nx + ny, p_open=0.1, p_solid=p_solid,
                              log10_k_range=(-2, 1))
    case = Case(nx, ny, tau=0.8, G=g, walls=walls, pressure=pressure and nx >= 3, rho_in=1.0005,
                rho_out=0.9995, forchheimer=1, medium=med, kn_beta=beta)
    s = gpu_sim(case, storage)
    s.step(steps)
    return s, (slice(1, -1) if walls else slice(None))


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_sums_match_the_fields(nx, ny, storage):
    for beta, pressure in ((0.0, False), (50.0, True)):
        s, fr = _sim(nx, ny, storage, beta, pressure)
        rho, ux, uy = (_np(t) for t in s.macroscopic())
        if fr != slice(None):
            assert not rho[0].any() and not rho[-1].any() and not ux[0].any() and not uy[-1].any()
        n = rho[fr].size
        _, um = s.permeability()
        # a thread's FP32-pair sums are good to ~2^-44, the FP64 ones to n 2^-53
        scale = np.abs(ux[fr]).mean()
        assert abs(um - ux[fr].mean()) <= 1e-12 * scale
        assert s.mass() == pytest.approx(rho[fr].sum(), rel=2e-7 if storage else 1e-7, abs=0)
        assert s.residual() == pytest.approx(1.0, rel=1e-12)
        s.step(2)
        _, vx, vy = (_np(t) for t in s.macroscopic())
        want = np.sqrt(((vx - ux)[fr] ** 2 + (vy - uy)[fr] ** 2).sum()
                       / (vx[fr] ** 2 + vy[fr] ** 2).sum())
        assert s.residual() == pytest.approx(want, rel=1e-11, abs=0)
        assert n == s.info().fluid_nodes
        s.close()


@pytest.mark.parametrize("nx,ny", SIZES)
def test_populations_and_permeability_are_exact(nx, ny):
    """Periodic lattice, rho0 = 1: a loaded state is d = fl32(f - w), read back
    as the FP64 w + d; k_a is the FP64 reciprocal of an FP32 number."""
    med = media.random_medium(nx, ny, seed=3, p_open=0.1, log10_k_range=(-4, 3))
    s = gpu_sim(Case(nx, ny, tau=0.8, medium=med), 0)
    f0 = media.random_populations(nx, ny, seed=3, base=W, amp=2e-3)
    f0[:, 0, 0] = W          # d = 0
    f0[0, -1, -1] += 3.0     # a value that carries into the next binade
    f0[1, -1, -1] -= 0.5     # and a negative sum
    s.set_populations(f0)
    w = W[:, None, None]
    want = w + (f0 - w).astype(np.float32).astype(np.float64)
    assert np.array_equal(_np(s.populations()), want)
    ka = _np(s.apparent_permeability())
    inv = (1.0 / ka).astype(np.float32).astype(np.float64)
    with np.errstate(divide="ignore"):
        assert np.array_equal(ka, 1.0 / inv)
    assert np.isinf(ka).any() == bool(np.isinf(med.k_i).any())
    s.close()


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("nbins", [1, 7, 64])
@pytest.mark.parametrize("g,p_solid", [(2e-5, 0.1), (1e-24, 0.1), (2e-5, 1.0)])
def test_histogram_replay(storage, nbins, g, p_solid):
    """Ordinary speeds, speeds below the range of the FP32 estimates, no flow."""
    for nx, ny in ((257, 40), (64, 613)):
        s, fr = _sim(nx, ny, storage, g=(g, 0.3 * g), p_solid=p_solid, steps=30)
        _, ux, uy = (_np(t)[fr] for t in s.macroscopic())
        sp = np.sqrt(ux * ux + uy * uy)
        um = sp.max()
        k = np.zeros(sp.shape, int) if um == 0.0 else \
            np.minimum(np.floor(sp / um * nbins), nbins - 1).astype(int)
        counts, got = s.velocity_histogram(nbins)
        assert got == um
        assert np.array_equal(counts, np.bincount(k.ravel(), minlength=nbins))
        s.close()
