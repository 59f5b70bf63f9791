"""Free directions on meshes away from the origin, small, large, torn and under a stale tree.

As in test_gpu_free_directions.py the reference is each view in a call of its own, too small to use them: images, path
signatures and ray counts must be equal bitwise. Where they can answer rays, fewer nodes are fetched, which says that they
were used.
"""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2012_03939_gb300 import scenes as S
from tests.test_gpu_bvh_builders import st  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


def _views(closed, at, scale, **kw):
    """Enough paths for free directions in one call (2^19 on a closed mesh, 2^21 on another), too few in each view's own."""
    if closed:
        vs = S.fibonacci_views(2, [131, 128], [128, 111], [16, 20])
    else:
        vs = S.fibonacci_views(6, [131, 128, 97, 128, 150, 131], [128, 111, 160, 128, 99, 128], [24, 24, 30, 24, 24, 24])
    for v in vs:
        v.eye, v.target = (tuple(np.asarray(x, np.float64) * scale + at) for x in (v.eye, v.target))
    return [dataclasses.replace(v, **kw) for v in vs]


def _equal_to_small_calls(st, scene, sc, B=4, seed=5):
    """One call over all views against a call per view; node fetches of both."""
    count = st.make_opts(count_visits=1)
    scene.backward(sc.views, B, seed, torch.zeros((sc.n_pixels, 3), device="cuda"))   # has them built on rough meshes too
    sig = torch.zeros(sc.n_pixels, dtype=torch.int64, device="cuda")
    img = scene.render(sc.views, B, seed, count, signatures=sig).cpu().numpy()
    many, few = scene.stats(), dict.fromkeys(("extension_rays", "shadow_rays", "node_visits", "shadow_node_visits"), 0)
    assert many["device_error"] == 0
    for v in sc.views:
        assert v.width * v.height * v.spp < 1 << 19
        s1, ref = torch.zeros_like(sig), torch.zeros((sc.n_pixels, 3), device="cuda")
        scene.render([v], B, seed, count, out=ref, signatures=s1)
        a, b = v.pixel_offset, v.pixel_offset + v.width * v.height
        np.testing.assert_array_equal(img[a:b], ref[a:b].cpu().numpy())
        np.testing.assert_array_equal(sig[a:b].cpu().numpy(), s1[a:b].cpu().numpy())
        s = scene.stats()
        assert s["device_error"] == 0
        for k in few:
            few[k] += s[k]
    assert (many["extension_rays"], many["shadow_rays"]) == (few["extension_rays"], few["shadow_rays"])
    return many, few


def _scene(V, F, views, rng, **kw):
    return S.Scene("free", S._f32(V), np.ascontiguousarray(F, np.int32), S.random_face_params(rng, len(F)),
                   env=S.lognormal_env(rng, 64, 32), views=views, max_bounces=4, **kw)


@pytest.mark.parametrize("mesh", ["sphere", "rough", "knot"])
@pytest.mark.parametrize("where,scale", [(10.0, 1.0), (100.0, 1.0), (1000.0, 1.0), (100.0, 0.05), (0.0, 1e-3), (0.0, 40.0),
                                         (0.0, 1e3)])
def test_moved_and_scaled_meshes(st, mesh, where, scale):  # noqa: F811
    rng = np.random.default_rng(7)
    if mesh == "sphere":
        V, F = S.icosphere(4)
        V = S.sinusoid_displace(V, rng, amp=0.3)
    elif mesh == "rough":
        V, F = S.uv_sphere(60, 31)
        V = S.fractal_displace(V, rng, amp=0.12)
    else:
        V, F = S.torus_knot(2, 3, 120, 12)   # 2880 faces: 190 paths each, a concave mesh uses them from 140 on
    at = where * np.array([1.0, -0.7, 0.4])
    sc = _scene(V * scale + at, F, _views(True, at, scale), rng)
    scene = st.Scene.from_scene(sc)
    many, few = _equal_to_small_calls(st, scene, sc)
    if (where, scale) in ((10.0, 1.0), (100.0, 0.05)):   # longest edges below a unit, vertices near enough to their faces
        assert many["node_visits"] + many["shadow_node_visits"] < 0.97 * (few["node_visits"] + few["shadow_node_visits"])
    scene.close()


def _torn(name, rng):
    if name == "soup":
        c = rng.uniform(-0.8, 0.8, (400, 1, 3))
        V = (c + rng.normal(size=(400, 3, 3)) * rng.uniform(0.02, 0.3, (400, 1, 1))).reshape(-1, 3)
        return V, np.arange(len(V)).reshape(-1, 3)
    if name == "unwelded":      # every face with vertices of its own
        V, F = S.icosphere(3)
        V = S.sinusoid_displace(V, rng, amp=0.3)[F.ravel()]
        return V, np.arange(len(V)).reshape(-1, 3)
    # two strips folded along x = 0 whose borders meet there with different subdivisions
    def strip(n, x, z):
        y = np.linspace(-0.9, 0.9, n + 1)
        V = np.concatenate([np.c_[0 * y, y, 0 * y], np.c_[0 * y + x, y, 0 * y + z]])
        i = np.arange(n)
        F = np.concatenate([np.c_[i, i + 1, i + n + 1], np.c_[i + 1, i + n + 2, i + n + 1]])
        return V, F if x > 0 else F[:, [0, 2, 1]]
    (V, F), (W, G) = strip(8, 0.9, 0.05), strip(13, -0.9, 0.3)
    return np.concatenate([V, W]), np.concatenate([F, G + len(V)])


@pytest.mark.parametrize("name", ["soup", "unwelded", "strips"])
@pytest.mark.parametrize("where", [0.0, 30.0])
def test_torn_meshes(st, name, where):  # noqa: F811
    rng = np.random.default_rng(11)
    V, F = _torn(name, rng)
    at = where * np.array([1.0, -0.7, 0.4])
    sc = _scene(V + at, F, _views(False, at, 1.0), rng)
    scene = st.Scene.from_scene(sc)
    many, few = _equal_to_small_calls(st, scene, sc)
    if name == "unwelded" and not where:
        assert many["shadow_node_visits"] < 0.9 * few["shadow_node_visits"]
    scene.close()


def test_deformed_under_a_stale_tree(st):  # noqa: F811
    """A refit keeps the topology: after a strong twist its boxes overlap, and the node records are built over them."""
    rng = np.random.default_rng(3)
    V, F = S.icosphere(4)
    sc = _scene(V, F, _views(True, 0.0, 1.0), rng)
    scene = st.Scene.from_scene(sc)
    a = 3.0 * V[:, 1:2]
    W = np.concatenate([V[:, :1] * np.cos(a) - V[:, 2:] * np.sin(a), V[:, 1:2],
                        V[:, :1] * np.sin(a) + V[:, 2:] * np.cos(a)], 1) * [1.3, 0.4, 0.8]
    scene.refit(torch.from_numpy(S._f32(W)).cuda())
    _equal_to_small_calls(st, scene, sc)
    scene.close()
