"""Contexts on several GPUs of one process (a context belongs to the device
that is current when it is created): kernels that need more than the default
48 KB of shared memory run on each of them, and a failure to raise the limit
is not kept.  Host logic, against a runtime without a GPU."""
import pytest

import fake_device as fake
from paper_1411_7051_gb300 import lbmp


@pytest.fixture()
def L(tmp_path):   # a fresh library: nothing left over from another test
    return fake.load(tmp_path)


LATTICES = [(64, 33, {}), (400, 400, dict(kn_beta=100.0)), (200, 200, dict(forchheimer=0)),
            (200, 200, dict(storage=1)), (200, 200, dict(storage=1, fp16_rounding=1, kn_beta=100.0)),
            (600, 500, dict(storage=1)), (1024, 1024, {}), (1100, 1024, dict(kn_beta=100.0)),
            (1100, 1024, dict(kn_beta=100.0, forchheimer=0)), (1100, 1024, dict(storage=1)),
            (300, 300, dict(storage=1, kernel=lbmp.KERNEL_STAGED))]


def test_lattices_step_on_every_device(L):
    for dev in (0, 1, 0):
        for nx, ny, kw in LATTICES:
            L.fake_set_device(dev)
            st, h = fake.create(L, fake.params(nx, ny, **kw))
            assert st == lbmp.OK
            L.fake_set_device(1 - dev)   # the context's device is not the caller's
            assert L.lbmp_step(h, 45) == lbmp.OK, (dev, nx, ny, kw, L.lbmp_last_error())
            assert L.fake_device() == 1 - dev
            L.lbmp_destroy(h)


@pytest.mark.parametrize("storage,rounding", [(0, 0), (1, 0), (1, 1)])
def test_batches_step_on_every_device(L, storage, rounding):
    p = fake.params(1, 1, storage=storage, fp16_rounding=rounding)
    for dev in (0, 1):
        for sizes in ([(64, 40), (256, 64)], [(1024, 600), (512, 1024)], [(48, 48)]):
            L.fake_set_device(dev)
            st, h = fake.create_batch(L, p, sizes)
            assert st == lbmp.OK
            for shape in range(10):
                assert L.lbmp_batch_set_shape(h, shape) == lbmp.OK
                for n in (3, 40):
                    assert L.lbmp_batch_step(h, n) == lbmp.OK, (dev, sizes, shape)
            L.lbmp_batch_destroy(h)


def test_failure_is_not_kept(L):
    """Every limit raised on the way fails once: the call reports it, the
    next lattice or batch of the kind works."""
    def lattice(p):
        st, h = fake.create(L, p)
        st = st or L.lbmp_step(h, 45)
        L.lbmp_destroy(h) if h else None
        return st

    def batch(p):
        st, h = fake.create_batch(L, p, [(256, 64)])
        st = st or L.lbmp_batch_set_shape(h, 9) or L.lbmp_batch_step(h, 3)
        L.lbmp_batch_destroy(h) if h else None
        return st

    kinds = [(lattice, fake.params(nx, ny, **kw)) for nx, ny, kw in LATTICES]
    kinds += [(batch, fake.params(1, 1, storage=s)) for s in (0, 1)]
    for run, p in kinds:
        L.fake_fail_attributes(100)
        assert run(p) == lbmp.ECUDA
        L.fake_fail_attributes(0)
        assert run(p) == lbmp.OK, L.lbmp_last_error()
