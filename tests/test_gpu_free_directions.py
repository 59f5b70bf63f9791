"""Free directions of a face (st_horizon.cuh): rays they answer are exactly rays that hit nothing.

A call of many paths builds per face the cells of directions in which other geometry may stand; its shading
kernel then neither traces nor queues rays that leave through an empty cell. The reference is the same views, each
in a call of its own too small to use them: images, path signatures and ray counts must be equal bitwise, whatever the mesh (open, closed, wound inward, rough, with
slivers, with several components, of one or two faces), the lights and the shading options.
"""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2012_03939_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def st():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2012_03939_gb300 import build
    build.build()
    from paper_2012_03939_gb300 import st as _st
    _st.lib()
    return _st


def _mesh(name, rng):
    """Vertices, faces."""
    if name in ("sphere", "inward", "two_spheres", "scaled"):
        V, F = S.icosphere(3)
        V = S.sinusoid_displace(V, rng, amp=0.3)
        if name == "inward":
            F = F[:, [0, 2, 1]]
        if name == "two_spheres":   # not one surface; each stands over the other's horizon
            F = np.concatenate([F, F + len(V)])
            V = np.concatenate([0.45 * V - [0.5, 0, 0], 0.45 * V + [0.5, 0.1, 0]])
        if name == "scaled":        # longest edges far above the hit distance bound's scale
            V = V * [1.5, 0.2, 0.9]
        return V, F
    if name == "rough":
        V, F = S.uv_sphere(60, 31)
        return S.fractal_displace(V, rng, amp=0.4), F
    if name == "slivers":           # poles of a fine sphere: faces a hundred times longer than wide
        return S.uv_sphere(400, 9)
    if name == "knot":
        return S.torus_knot(2, 3, 120, 16)
    if name == "one_face":
        return np.array([[-0.9, -0.8, 0.0], [0.9, -0.7, 0.1], [0.0, 0.9, -0.1]]), np.array([[0, 1, 2]], np.int32)
    if name == "two_faces":         # a valley
        return (np.array([[0, -0.9, 0.0], [0, 0.9, 0.0], [-0.9, 0, 0.5], [0.9, 0, 0.5]]),
                np.array([[0, 1, 2], [1, 0, 3]], np.int32))
    sc = S.color_bleed(n=6)
    return sc.vertices - 0.5, sc.faces


CASES = [(m, light, smooth) for m in ("sphere", "inward", "two_spheres", "scaled", "rough", "slivers", "knot",
                                      "one_face", "two_faces", "planes")
         for light, smooth in (("env", False), ("points+env", True))]


@pytest.mark.parametrize("mesh,light,smooth", CASES)
def test_free_directions_change_nothing(st, mesh, light, smooth):
    rng = np.random.default_rng(len(mesh) + 17 * smooth)
    V, F = _mesh(mesh, rng)
    lights = S._f32([[2.0, 1.5, 2.5], [-0.3, 3.0, 0.2]]) if "points" in light else np.zeros((0, 3), np.float32)
    views = S.fibonacci_views(6, [131, 128, 97, 128, 150, 131], [128, 111, 160, 128, 99, 128], [24, 24, 30, 24, 24, 24])
    closed = mesh not in ("two_spheres", "one_face", "two_faces", "planes")
    if closed:   # used from 2^19 paths on; below 5 * 2^17 every first ray goes through the tree in both
        views = [dataclasses.replace(v, spp=s) for v, s in zip(views, (16, 20))]
    sc = S.Scene("free", S._f32(V), np.ascontiguousarray(F, np.int32), S.random_face_params(rng, len(F)),
                 light_pos=lights, light_intensity=np.full_like(lights, 5.0), env=S.lognormal_env(rng, 64, 32),
                 views=views, max_bounces=4, smooth_normals=smooth)
    scene = st.Scene.from_scene(sc)
    sig = torch.zeros(sc.n_pixels, dtype=torch.int64, device="cuda")
    # an adjoint builds them on rough and concave meshes too, where a forward call alone would not
    scene.backward(sc.views, 4, 5, torch.zeros((sc.n_pixels, 3), device="cuda"))
    img = scene.render(sc.views, 4, 5, signatures=sig).cpu().numpy()
    stats = scene.stats()
    paths = sum(v.width * v.height * v.spp for v in views)
    assert 1 << 19 <= paths < 5 << 17 if closed else paths >= 1 << 21   # enough paths to use them
    assert stats["device_error"] == 0
    ext = shadow = 0
    for v in views:
        assert v.width * v.height * v.spp < 1 << 19
        s1 = torch.zeros(sc.n_pixels, dtype=torch.int64, device="cuda")
        ref = torch.zeros((sc.n_pixels, 3), device="cuda")
        scene.render([v], 4, 5, out=ref, signatures=s1)
        a, b = v.pixel_offset, v.pixel_offset + v.width * v.height
        np.testing.assert_array_equal(img[a:b], ref[a:b].cpu().numpy())
        np.testing.assert_array_equal(sig[a:b].cpu().numpy(), s1[a:b].cpu().numpy())
        s = scene.stats()
        assert s["device_error"] == 0
        ext += s["extension_rays"]
        shadow += s["shadow_rays"]
    assert (stats["extension_rays"], stats["shadow_rays"]) == (ext, shadow)
    scene.close()


def test_free_directions_skip_the_tree_on_a_convex_mesh(st):
    """On a smooth convex mesh nearly every bounce and environment ray is answered without a node fetch, and a
    vertex update discards what was built."""
    sc = S.make("edges", n_views=8)
    sc.env = S.lognormal_env(np.random.default_rng(3), 64, 32)
    scene = st.Scene.from_scene(sc)
    o = st.make_opts(count_visits=1)
    scene.render(sc.views, 3, 1, o)
    s = scene.stats()
    assert s["shadow_node_visits"] < 0.5 * s["shadow_rays"]
    V = scene.vertices.clone()
    V[:, 0] *= 0.8
    scene.refit(V)
    img = scene.render(sc.views, 3, 1).cpu().numpy()
    fresh = st.Scene.from_scene(sc, vertices=V.cpu())
    np.testing.assert_array_equal(img, fresh.render(sc.views, 3, 1).cpu().numpy())
    scene.close()
    fresh.close()


@pytest.mark.parametrize("mesh", ["sphere", "rough", "knot"])
def test_lists_of_calls_below_a_million_rays_equal_the_tree(st, mesh):
    """From 5 * 2^17 rays on a closed mesh's first rays are found in lists that keep its back faces: the same hits as
    the tree's, at silhouettes too."""
    V, F = _mesh(mesh, np.random.default_rng(8))
    rng = np.random.default_rng(9)
    views = S.fibonacci_views(4, [200, 129, 181, 97], [131, 177, 120, 210], [9, 9, 9, 8])
    sc = S.Scene("lists", S._f32(V), np.ascontiguousarray(F, np.int32), S.random_face_params(rng, len(F)),
                 env=S.lognormal_env(rng, 64, 32), views=views, max_bounces=2)
    paths = sum(v.width * v.height * v.spp for v in views)
    assert 5 << 17 <= paths < 1 << 20 and 4 * len(F) * len(views) <= paths
    scene = st.Scene.from_scene(sc)
    sig = torch.zeros(sc.n_pixels, dtype=torch.int64, device="cuda")
    img = scene.render(views, 2, 11, st.make_opts(count_visits=1), signatures=sig)
    many = scene.stats()
    visits = 0
    ref, s1 = torch.zeros_like(img), torch.zeros_like(sig)
    for v in views:
        scene.render([v], 2, 11, st.make_opts(count_visits=1), out=ref, signatures=s1)
        visits += scene.stats()["node_visits"]
    assert many["node_visits"] < 0.5 * visits   # the lists were used
    np.testing.assert_array_equal(sig.cpu().numpy(), s1.cpu().numpy())
    np.testing.assert_array_equal(img.cpu().numpy(), ref.cpu().numpy())
    scene.close()
