"""Primary lists of coarse meshes: a warp takes few of their faces, whose cells it goes through together.

A closed mesh's call of 5 * 2^17 rays builds lists (test_gpu_free_directions.py compares meshes of many faces); here few faces
cover many cells each, at every number of faces a warp can take, and the tree's hits are the reference: each view in a
call of its own, too small to build lists. With next to no faces the call does without lists.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2012_03939_gb300 import scenes as S
from tests.test_gpu_bvh_builders import st  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


def _scene(subdiv, n_views, rng):
    V, F = S.icosphere(subdiv)
    V = S.sinusoid_displace(V, rng, amp=0.2)
    w = int(np.sqrt(700000 / n_views / 8))
    views = S.fibonacci_views(n_views, [w + k % 3 for k in range(n_views)], [w - k % 2 for k in range(n_views)], [8] * n_views)
    paths = sum(v.width * v.height * v.spp for v in views)
    assert 5 << 17 <= paths < 1 << 20 and 4 * len(F) * n_views <= paths
    return S.Scene("coarse", S._f32(V), np.ascontiguousarray(F, np.int32), S.random_face_params(rng, len(F)),
                   env=S.lognormal_env(rng, 64, 32), views=views, max_bounces=2)


@pytest.mark.parametrize("subdiv,n_views,lists", [(0, 2, False), (0, 30, True), (1, 7, True), (2, 2, True), (2, 16, True),
                                                  (3, 4, True), (3, 16, True), (4, 4, True), (4, 16, True)])
def test_lists_of_coarse_meshes_equal_the_tree(st, subdiv, n_views, lists):  # noqa: F811
    sc = _scene(subdiv, n_views, np.random.default_rng(subdiv + 10 * n_views))
    scene = st.Scene.from_scene(sc)
    count = st.make_opts(count_visits=1)
    sig, s1 = (torch.zeros(sc.n_pixels, dtype=torch.int64, device="cuda") for _ in range(2))
    img = scene.render(sc.views, 2, 11, count, signatures=sig)
    many, visits, ref = scene.stats(), 0, torch.zeros_like(img)
    for v in sc.views:
        assert v.width * v.height * v.spp < 5 << 17
        scene.render([v], 2, 11, count, out=ref, signatures=s1)
        s = scene.stats()
        assert s["device_error"] == 0
        visits += s["node_visits"]
    assert many["device_error"] == 0 and (many["node_visits"] < 0.7 * visits) == lists
    np.testing.assert_array_equal(sig.cpu().numpy(), s1.cpu().numpy())
    np.testing.assert_array_equal(img.cpu().numpy(), ref.cpu().numpy())
    scene.close()
