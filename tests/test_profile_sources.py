"""The hashes that tie committed ncu figures to their kernels cover every source
that the kernels are made of: a change of any of them must make the figures
stale (tests/test_profiles.py)."""
import os
import re

import pytest

from paper_1411_7051_gb300 import build


def _device_headers(name, seen):
    """The .cuh files that a source includes, directly or through another."""
    with open(os.path.join(build.CSRC, name)) as fh:
        for inc in re.findall(r'^#include "(\w+\.\w+)"', fh.read(), re.M):
            if inc not in seen and os.path.exists(os.path.join(build.CSRC, inc)):
                seen.add(inc)
                _device_headers(inc, seen)
    return {h for h in seen if h.endswith(".cuh")}


@pytest.mark.parametrize("files,units", [
    (build.STEP_KERNEL_FILES, ["kernels.cu", "fused.cu", "tile.cu"]),
    # the recompute of a gradient runs the step kernels
    (build.ADJOINT_KERNEL_FILES, ["adjoint.cu", "kernels.cu", "fused.cu"]),
    (build.BATCH_KERNEL_FILES, ["batch.cu"])])
def test_hashed_files_cover_the_kernels(files, units):
    need = set(units)
    for unit in units:
        need |= _device_headers(unit, set())
    assert need <= set(files), sorted(need - set(files))
    assert set(files) <= set(build.SOURCES + build.HEADERS)
