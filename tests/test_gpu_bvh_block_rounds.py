"""The rounds and levels of a tree build that one block runs by itself: the last ones of the clustering (at most 1024
clusters) and those of the 4-wide collapse with at most 1024 entries. Sizes on both sides of either limit, from two faces
on; the hits of the radix tree, whose build shares the collapse alone, are the reference for the clustering's.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2012_03939_gb300 import scenes as S
from tests.test_gpu_bvh_builders import _check_tree, _tree, st  # noqa: F401  (st: the fixture)

pytestmark = pytest.mark.gpu


def _soup(n, seed):
    """n disjoint-vertex triangles of mixed sizes."""
    rng = np.random.default_rng(seed)
    c = rng.uniform(-1, 1, (n, 1, 3))
    return S._f32((c + rng.normal(size=(n, 3, 3)) * rng.uniform(0.01, 0.2, (n, 1, 1))).reshape(-1, 3))


@pytest.mark.parametrize("n", [2, 3, 17, 1023, 1024, 1025, 2600, 9001])
def test_trees_around_a_block_of_clusters(st, n):  # noqa: F811
    rng = np.random.default_rng(n)
    F = np.arange(3 * n, dtype=np.int32).reshape(n, 3)
    d = rng.normal(size=(4096, 3))
    rays = np.c_[rng.uniform(-1.5, 1.5, (4096, 3)), np.zeros(4096), d / np.linalg.norm(d, axis=1, keepdims=True),
                 np.full(4096, 1e30)].astype(np.float32)
    rays = torch.from_numpy(rays).cuda()
    sc = S.Scene("soup", _soup(n, 1), F, S.random_face_params(rng, n), light_pos=S._f32([[3, 3, 3]]),
                 light_intensity=S._f32([[1, 1, 1]]), views=S.fibonacci_views(2, [16, 16], [16, 16], [1, 1]), max_bounces=1)
    V2 = _soup(n, 2)
    hits = {}
    for b in ("ploc", "lbvh"):
        scene = st.Scene.from_scene(sc, bvh_builder=b)
        out = [x.cpu().numpy() for x in scene.trace_closest(rays)]
        scene.rebuild(torch.from_numpy(V2).cuda())
        _check_tree(*_tree(scene), V2, F)
        out += [x.cpu().numpy() for x in scene.trace_closest(rays)]
        assert scene.stats()["device_error"] == 0
        hits[b] = out
        scene.close()
    for x, y in zip(hits["ploc"], hits["lbvh"]):
        np.testing.assert_array_equal(x, y)
