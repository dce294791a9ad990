"""The accesses that put a whole vector together off the 16-byte grid (jb_offgrid.h), run on
the host: each byte of the vector once and no other one, which another thread may be writing,
aligned for its size, and the right bits."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def accesses():
    from paper_2306_10015_gb300 import build
    src = os.path.join(ROOT, "tests", "helpers", "off_grid.cpp")
    out_dir = os.path.join(ROOT, "tests", "_build")
    os.makedirs(out_dir, exist_ok=True)
    out = os.path.join(out_dir, f"liboff_grid.{os.getpid()}.so")
    subprocess.run([build.nvcc(), "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC, src, "-o", out],
                   check=True)
    lib = ctypes.CDLL(out)
    os.remove(out)
    for f in (lib.off_grid_load, lib.off_grid_store):
        f.argtypes = [ctypes.c_void_p, ctypes.c_uint64, ctypes.c_uint32, ctypes.c_void_p, ctypes.c_void_p]
    return lib


@pytest.mark.parametrize("at,align", [(8, 8), (24, 8), (4, 4), (12, 4), (2, 2), (6, 2), (14, 2)])
def test_touches_its_own_bytes_once(accesses, at, align):
    rng = np.random.default_rng(at)
    whole = rng.integers(0, 256, 64).astype(np.uint8)
    own = np.zeros(64, dtype=np.int32)
    own[at:at + 16] = 1

    buf, got, reads = whole.copy(), np.zeros(4, dtype=np.uint32), np.zeros(64, dtype=np.int32)
    assert accesses.off_grid_load(buf.ctypes.data, at, align, got.ctypes.data, reads.ctypes.data) == 0
    assert np.array_equal(reads, own)
    assert np.array_equal(got.view(np.uint8), whole[at:at + 16])

    new, writes = rng.integers(0, 1 << 32, 4, dtype=np.uint64).astype(np.uint32), np.zeros(64, dtype=np.int32)
    assert accesses.off_grid_store(buf.ctypes.data, at, align, new.ctypes.data, writes.ctypes.data) == 0
    assert np.array_equal(writes, own)
    want = whole.copy()
    want[at:at + 16] = new.view(np.uint8)
    assert np.array_equal(buf, want)
