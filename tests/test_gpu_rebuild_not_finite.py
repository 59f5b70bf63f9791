"""A rebuild at vertices that are not finite fails and leaves the scene usable.

The clustering's boxes are not finite then, no round merges two of them, and every cluster is kept: all n of them are
written to the round's output before the host reads that nothing merged. That output is the scene's own memory.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2012_03939_gb300 import scenes as S
from tests.test_gpu_bvh_builders import st  # noqa: F401  (the fixture)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_scratch_holds_every_cluster(tmp_path):
    """Three arrays of n boxes, apart from one another and within the allocation, which also holds 3 records a node."""
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "check.cu"
    src.write_text('''#include "st_internal.h"
constexpr bool fits(size_t n) {
  constexpr auto apart = [](size_t a, size_t b, size_t n) { return a + n <= b || b + n <= a; };
  const st::PlocScratch p = st::ploc_scratch(n);
  return apart(p.lo1, p.hi0, n) && apart(p.lo1, p.hi1, n) && apart(p.hi0, p.hi1, n) && p.lo1 + n <= p.records &&
         p.hi0 + n <= p.records && p.hi1 + n <= p.records && 3 * (n > 1 ? n - 1 : 1) <= p.records;
}
static_assert(fits(1) && fits(2) && fits(1025) && fits(1000000) && fits(3000000000ull), "clusters past the scratch");
''')
    subprocess.run([nvcc, "-std=c++17", "-c", str(src), "-o", str(tmp_path / "check.o"),
                    "-I" + os.path.join(ROOT, "paper_2012_03939_gb300", "csrc"), "-I" + os.path.join(ROOT, "include")],
                   check=True, capture_output=True, timeout=600)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [2, 1024, 1025, 5000])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_rebuild_at_bad_vertices_fails_and_the_next_succeeds(st, n, bad):  # noqa: F811
    rng = np.random.default_rng(n)
    V = S._f32(rng.uniform(-1, 1, (n, 1, 3)) + 0.1 * rng.normal(size=(n, 3, 3))).reshape(-1, 3)
    F = np.arange(3 * n, dtype=np.int32).reshape(n, 3)
    sc = S.Scene("soup", V, F, S.random_face_params(rng, n), light_pos=S._f32([[3, 3, 3]]), light_intensity=S._f32([[1, 1, 1]]),
                 views=S.fibonacci_views(1, [16], [16], [1]), max_bounces=1)
    d = rng.normal(size=(4096, 3))
    rays = torch.from_numpy(np.c_[rng.uniform(-1.5, 1.5, (4096, 3)), np.zeros(4096),
                                  d / np.linalg.norm(d, axis=1, keepdims=True), np.full(4096, 1e30)].astype(np.float32)).cuda()
    scene = st.Scene.from_scene(sc)
    ref = [x.cpu().numpy() for x in scene.trace_closest(rays)]
    with pytest.raises(st.StError):
        scene.rebuild(torch.full((3 * n, 3), bad, device="cuda"))
    scene.rebuild(torch.from_numpy(V).cuda())
    for a, b in zip(scene.trace_closest(rays), ref):
        np.testing.assert_array_equal(a.cpu().numpy(), b)
    assert scene.stats()["device_error"] == 0
    scene.close()
