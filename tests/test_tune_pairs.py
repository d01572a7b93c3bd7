"""The batch autotuner and the two-step launches beside its staged candidate: a
shape tuned with them serves no batch without them, nor the reverse, and the
tuner times them whatever the number of steps.  Host logic, against a runtime
without a GPU (a launch takes a millisecond there)."""
import ctypes

import pytest

import fake_device as fake
from paper_1411_7051_gb300 import lbmp

PAIRS = [(256, 256)] * 8                       # two pairs of nodes a lane from 10^6 nodes on
PAIRS2 = [(1024, 1024)] * 2
NARROW = [(256, 256)] * 7 + [(48, 300), (256, 200)]   # same class as PAIRS, no pairs
NARROW2 = [(1024, 1024)] * 2 + [(48, 48)]
STAGED = 9


@pytest.fixture()
def L(tmp_path):   # a fresh library: an empty cache
    return fake.load(tmp_path)


def _tune(L, sizes, steps=4):
    st, h = fake.create_batch(L, fake.params(1, 1), sizes)
    assert st == lbmp.OK
    shape, ms, hit = ctypes.c_int32(), ctypes.c_double(), ctypes.c_int32()
    assert L.lbmp_batch_tune_cached(h, steps, ctypes.byref(shape), ctypes.byref(ms),
                                    ctypes.byref(hit)) == lbmp.OK
    L.lbmp_batch_destroy(h)
    return shape.value, hit.value


@pytest.mark.parametrize("pairs,narrow", [(PAIRS, NARROW), (PAIRS2, NARROW2)])
@pytest.mark.parametrize("pairs_first", [True, False])
def test_batches_with_and_without_pairs_are_tuned_apart(L, tmp_path, monkeypatch, pairs, narrow,
                                                        pairs_first):
    path = tmp_path / "tune.txt"
    monkeypatch.setenv("LBMP_TUNE_CACHE", str(path))
    cfg = lbmp.SimConfig(1, 1, bc_x=lbmp.BCX_PRESSURE, bc_y=lbmp.BCY_WALLS, forchheimer=1)
    key = lbmp.batch_class(cfg, pairs, 152)
    assert key == lbmp.batch_class(cfg, narrow, 152)
    order = (pairs, narrow) if pairs_first else (narrow, pairs)
    for sizes in order:
        assert _tune(L, sizes) == (STAGED if sizes is pairs else 0, 0)
    for sizes in order:
        assert _tune(L, sizes) == (STAGED if sizes is pairs else 0, 1)
    lines = [line.split()[:2] for line in path.read_text().splitlines()]
    assert [key, "0"] in lines and len(lines) == 2
    # a line of a library that timed no pairs serves only batches without them
    L.lbmp_batch_tune_cache_clear()
    path.write_text(f"{key} 3 0.5\n")
    assert _tune(L, narrow) == (3, 1)
    assert _tune(L, pairs) == (STAGED, 0)


@pytest.mark.parametrize("steps", [1, 2, 3])
def test_the_tuner_times_pairs(L, steps):
    assert _tune(L, PAIRS2, steps) == (STAGED, 0)
