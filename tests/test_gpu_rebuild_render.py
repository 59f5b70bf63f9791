"""Renders and adjoints after a rebuild of the hierarchy: the 4-wide tree's node count changes with it.

A batched call is a captured graph that holds launch sizes and arguments as captured, the node count among them (the
traversal's bounds, and the build of the faces' free directions). After a rebuild to fewer and to more nodes the same
views must render what a scene created at those vertices renders.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2012_03939_gb300 import scenes as S
from tests.test_gpu_bvh_builders import st  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu

B, SEED = 3, 23


def _vertices(base, seed):
    """The base mesh with noise of the seed: rough, so that some rays are free and some hit."""
    rng = np.random.default_rng(seed)
    return S._f32(base * (1.0 + 0.004 * rng.normal(size=(len(base), 1))) + 0.3 * rng.normal(size=3))


def _step(scene, sc, w):
    dV, dF = scene.backward(sc.views, B, SEED, w, _opts())
    built = scene.stats()["kernel_launches"]
    scene.backward(sc.views, B, SEED, w, _opts())
    assert built - scene.stats()["kernel_launches"] == 6 + 3   # primary lists and free directions were built, and then kept
    sig = torch.zeros(sc.n_pixels, dtype=torch.int64, device="cuda")
    img = scene.render(sc.views, B, SEED, signatures=sig)
    s = scene.stats()
    assert s["device_error"] == 0
    return img.cpu().numpy(), sig.cpu().numpy(), dV.cpu().numpy(), dF.cpu().numpy(), s


def _opts():
    from paper_2012_03939_gb300 import st as m
    return m.make_opts(edge_term=1)


@pytest.mark.parametrize("builder", ["ploc", "lbvh"])
def test_calls_after_a_rebuild_to_fewer_and_to_more_nodes(st, builder):  # noqa: F811
    base, F = S.icosphere(4)
    rng = np.random.default_rng(1)
    sc = S.Scene("rebuilt", _vertices(base, 0), np.ascontiguousarray(F, np.int32), S.random_face_params(rng, len(F)),
                 env=S.lognormal_env(rng, 64, 32), max_bounces=B, views=S.fibonacci_views(4, [128] * 4, [128] * 4, [9] * 4))
    # enough paths for free directions (2^19 and 200 rays a face), in the forward and the adjoint
    assert 1 << 19 <= sum(v.width * v.height * v.spp for v in sc.views)
    w = torch.from_numpy(np.random.default_rng(2).normal(size=(sc.n_pixels, 3)).astype(np.float32)).cuda()
    probe = st.Scene.from_scene(sc, bvh_builder=builder)
    nodes = {}
    for k in range(1, 9):
        probe.rebuild(torch.from_numpy(_vertices(base, k)).cuda())
        nodes[k] = probe.stats()["bvh4_nodes"]
    probe.close()
    by = sorted(nodes, key=nodes.get)
    few, mid, many = by[0], by[4], by[-1]
    assert nodes[few] < nodes[mid] < nodes[many]
    scene = st.Scene.from_scene(sc, vertices=_vertices(base, mid), bvh_builder=builder)
    for k in (mid, few, many, few, mid):
        V = _vertices(base, k)
        scene.rebuild(torch.from_numpy(V).cuda())
        got = _step(scene, sc, w)
        assert got[4]["bvh4_nodes"] == nodes[k]
        fresh = st.Scene.from_scene(sc, vertices=V, bvh_builder=builder)
        ref = _step(fresh, sc, w)
        fresh.close()
        np.testing.assert_array_equal(got[0], ref[0])
        np.testing.assert_array_equal(got[1], ref[1])
        assert (got[4]["extension_rays"], got[4]["shadow_rays"]) == (ref[4]["extension_rays"], ref[4]["shadow_rays"])
        for a, b in zip(got[2:4], ref[2:4]):   # the scatter's FP32 atomics add in any order
            np.testing.assert_allclose(a, b, rtol=1e-4, atol=1e-5 * np.abs(b).max())
    scene.close()
