"""Runs a piece of Python in a process of its own in which libbvf sits on the
fake CUDA runtime of fake_cuda.c: whole calls of the C ABI on a machine
without a GPU, up to the launches, which run nothing.  For what the host side
decides: which kernels a call launches, what a failed allocation leaves
behind, when a recording is made anew."""
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = r"""
import ctypes, os, re
import numpy as np
from paper_2301_12727_gb300 import bvf, fno
L = bvf.lib()
fake = ctypes.CDLL(os.environ["LD_PRELOAD"])
fake.fake_log.restype = ctypes.c_char_p
fake.fake_free_mem.argtypes = [ctypes.c_size_t]
for f in ("fake_mallocs", "fake_malloc_bytes", "fake_instantiated", "fake_launches"):
    getattr(fake, f).restype = ctypes.c_longlong
OK, ARG, NOMEM = bvf.BVF_OK, bvf.BVF_E_ARG, bvf.BVF_E_NOMEM
WATER = [1000.0, 1500.0, 0.0, 0.0, 0.0, 0.6, 4178.0, 0.0, 1.0]
BONE = [1850.0, 2800.0, 1500.0, 85.0, 170.0, 0.32, 1313.0, 0.008, 0.16]
keep = []

def buf(n):
    b = ctypes.create_string_buffer(int(n))
    keep.append(b)
    return ctypes.cast(b, ctypes.c_void_p)

def create(nx, ny=8, nz=8, n_sls=2, storage=0, n_pml=2):
    g = bvf.Grid(nx, ny, nz, 0.5e-3, 4e-8, n_pml, 1e-3)
    ph = bvf.Physics(5e5, 1.0, n_sls, storage, 1e5)
    c = ctypes.c_void_p()
    rc = L.bvf_create(ctypes.byref(g), ctypes.byref(ph), ctypes.byref(c))
    return rc, c

def context(nx, ny=8, nz=8, table=(WATER,), **kw):
    rc, c = create(nx, ny, nz, **kw)
    assert rc == OK, L.bvf_last_error(None)
    materials(c, nx * ny * nz, table)
    return c

def materials(c, n, table):
    rc = L.bvf_set_materials(c, buf(n), bvf.material_array(list(table)), len(table))
    assert rc == OK, L.bvf_last_error(c)

def launches():
    # (kernel name, grid, dynamic shared memory) of every launch since the last call
    rows = [r.rsplit(" ", 4) for r in fake.fake_log().decode().splitlines()]
    fake.fake_log_clear()
    return [(re.search("k_[a-z0-9_]+", n).group(), (int(x), int(y), int(z)), int(s))
            for n, x, y, z, s in rows]

def launched():
    return [(n, s) for n, _, s in launches()]
"""


def run(code, tmp_path, **env):
    """Run `code` after PRELUDE; a failing assertion in it fails the test."""
    from paper_2301_12727_gb300 import build
    build.build()
    so = str(tmp_path / "libfakecuda.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-w", "-I/usr/local/cuda/include",
                    os.path.join(HERE, "fake_cuda.c"), "-o", so], check=True)
    e = {k: v for k, v in os.environ.items() if not k.startswith("BVF_")}
    e.update(LD_PRELOAD=so, PYTHONPATH=ROOT, **env)
    r = subprocess.run([sys.executable, "-c", PRELUDE + code], env=e, cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    return r.stdout
