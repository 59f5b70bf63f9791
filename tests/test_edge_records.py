"""The screen records of the edge candidates: every listed candidate has one, and one that is not drawable takes no sample.

The list counts an edge that one kernel's clip calls drawable; the kernel that writes the records clips it again, and where
the segment only touches the image the two may round differently. Such a place must not keep what the memory held before:
its edge number would index the vertices.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def trip(tmp_path_factory):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    out = str(tmp_path_factory.mktemp("edges") / "check.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                    os.path.join(HERE, "edge_record_check.cu"), "-o", out], check=True, capture_output=True, timeout=600)
    L = ctypes.CDLL(out)

    def f(drawable, e, vals, fill):
        src, dst, k = np.asarray(vals, np.float32), np.zeros(9, np.float32), ctypes.c_int()
        ok = L.edge_round_trip(int(drawable), int(e), src.ctypes.data_as(ctypes.c_void_p), ctypes.c_ubyte(fill),
                               dst.ctypes.data_as(ctypes.c_void_p), ctypes.byref(k))
        return bool(ok), dst, k.value
    return f


@pytest.mark.parametrize("fill", [0, 0x01, 0x7f, 0xff])
def test_candidates_that_are_not_drawable_take_no_sample(trip, fill):
    ok, vals, e = trip(False, 0, np.zeros(9), fill)
    assert not ok and e < 0
    np.testing.assert_array_equal(vals, 0)


@pytest.mark.parametrize("e", [0, 1, 12345, 2**31 - 1])
def test_drawable_candidates_are_read_back(trip, e):
    want = np.random.default_rng(e).normal(size=9).astype(np.float32)
    ok, vals, got = trip(True, e, want, 0xff)
    assert ok and got == e
    np.testing.assert_array_equal(vals, want)
