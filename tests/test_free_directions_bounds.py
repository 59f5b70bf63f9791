"""The bounds of the free directions (st_horizon.cuh) against the watertight test, on the host.

No ray that a face's cells call free may hit the triangle that marked them, wherever the pair lies: coordinates from one
to ten thousand, faces from a thousandth to one, neighbours that share an edge or a vertex, meet an edge between its ends
or stand near, at rises down to one rounding of the coordinates. horizon_check.cu holds the pairs and the rays.
"""
import ctypes
import os
import shutil
import subprocess
from concurrent.futures import ThreadPoolExecutor

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    out = str(tmp_path_factory.mktemp("horizon") / "check.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                    "-I" + os.path.join(os.path.dirname(HERE), "include"), os.path.join(HERE, "horizon_check.cu"), "-o", out],
                   check=True, capture_output=True, timeout=600)
    f = ctypes.CDLL(out).hz_check
    f.restype = ctypes.c_longlong
    f.argtypes = [ctypes.c_ulonglong, ctypes.c_longlong, ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_int,
                  ctypes.POINTER(ctypes.c_longlong)]
    return f


@pytest.mark.parametrize("where", [1.0, 10.0, 30.0, 100.0, 1000.0, 10000.0])
def test_no_free_ray_hits_the_neighbour(check, where):
    def one(job):
        kind, size = job
        out = (ctypes.c_longlong * 2)()
        wrong = check(1000 * kind + int(where), 200000, 8, where, size, kind, out)
        return job, wrong, out[0], out[1]

    jobs = [(kind, size) for kind in range(4) for size in (1e-3, 1e-2, 0.1, 1.0)]
    with ThreadPoolExecutor(8) as ex:
        got = list(ex.map(one, jobs))
    assert not [g for g in got if g[1]], [g for g in got if g[1]]
    if where < 1000.0:   # beyond, a vertex of these sizes lies too far off its face
        assert sum(g[3] for g in got) > 0.05 * sum(g[2] for g in got)   # rays were answered
