"""The library linked against a CUDA runtime that runs nothing
(fake_cudart.cpp): its host logic without a GPU."""
import ctypes
import os
import subprocess

import numpy as np

from paper_1411_7051_gb300 import build, lbmp

HERE = os.path.dirname(os.path.abspath(__file__))


def load(directory):
    """The library with the prototypes of ``lbmp.load``, built in directory."""
    build.build()
    objs = [os.path.join(build.OUT_DIR, n.replace(".cu", ".o")) for n in build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    out = os.path.join(str(directory), "liblbmp_fake.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-Wl,-Bsymbolic", "-I", include,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", out, "-ldl", "-lpthread"],
                   check=True)
    keep, lbmp._lib = lbmp._lib, None
    try:
        L = lbmp.load(out)
    finally:
        lbmp._lib = keep
    for f in (L.fake_launches, L.fake_blocks):
        f.restype = ctypes.c_longlong
        f.argtypes = [ctypes.c_char_p]
    L.fake_capture.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return L


def params(nx, ny, **kw):
    base = dict(bc_x=lbmp.BCX_PRESSURE, bc_y=lbmp.BCY_WALLS, rho_in=1.0005, rho_out=0.9995,
                forchheimer=1)
    base.update(kw)
    stream = base.pop("stream", None)
    return lbmp.SimConfig(nx, ny, **base).to_params(stream)


def create(L, p):
    """(status, handle) of a lattice with fields."""
    h = ctypes.c_void_p()
    st = L.lbmp_create(ctypes.byref(p), ctypes.byref(h))
    if st == lbmp.OK:
        f = np.ones(p.nx * p.ny).ctypes.data_as(ctypes.c_void_p)
        st = L.lbmp_set_fields(h, f, f, f, lbmp.DEVICE)
    return st, h


def create_batch(L, p, sizes):
    nx, ny = ((ctypes.c_int32 * len(sizes))(*v) for v in zip(*sizes))
    h = ctypes.c_void_p()
    st = L.lbmp_batch_create(ctypes.byref(p), len(sizes), nx, ny, ctypes.byref(h))
    for i in range(len(sizes)):
        f = np.ones(sizes[i][0] * sizes[i][1]).ctypes.data_as(ctypes.c_void_p)
        st = st or L.lbmp_batch_set_fields(h, i, f, f, f, lbmp.DEVICE)
    return st, h
