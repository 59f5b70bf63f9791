"""Which calls build the faces' free directions: both sides of each line of the rule.

A call that builds them enqueues three launches more than the same call repeated on the same vertices. The calls here have too
few paths for the primary lists (5 * 2^17 on a closed mesh), which would be built by the first call as well.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2012_03939_gb300 import scenes as S
from tests.test_gpu_bvh_builders import st  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu

PATHS = 4 * 128 * 128 * 9   # 589824: above 2^19


def _mesh(name):
    rng = np.random.default_rng(1)
    # the spheres cover 0.58 of a square view, the knots about 0.4
    if name == "smooth":            # every direction free but the lowest
        V, F = S.icosphere(5)       # 20480 faces: 16.7 hits each
        return S.sinusoid_displace(V, rng), F
    if name == "fine fractal":      # 25600 faces: 14 hits each
        V, F = S.uv_sphere(160, 81)
        return S.fractal_displace(V, np.random.default_rng(7)), F
    if name == "knot":              # 0.41 free; 3840 faces: 60 hits each
        return S.torus_knot(2, 3, 120, 16)
    if name == "small knot":        # 1536 faces: 150 hits each
        return S.torus_knot(2, 3, 128, 6)
    assert name == "rough"          # 0.3 free; 1600 faces: 290 hits each
    V, F = S.uv_sphere(40, 21)
    return S.fractal_displace(V, np.random.default_rng(7), amp=0.4), F


def _builds(st, mesh, light, B, scale, adjoint, w=128, h=128):
    V, F = _mesh(mesh)
    rng = np.random.default_rng(2)
    views = S.fibonacci_views(4, [w] * 4, [h] * 4, [9] * 4)
    if light == "view":
        views = S.with_view_lights(views)
    for v in views:
        v.eye, v.target = tuple(np.asarray(v.eye) * scale), tuple(np.asarray(v.target) * scale)
    sc = S.Scene("rule", S._f32(V * scale), np.ascontiguousarray(F, np.int32), S.random_face_params(rng, len(F)),
                 env=S.lognormal_env(rng, 64, 32) if light == "env" else None, views=views, max_bounces=B)
    assert sum(v.width * v.height * v.spp for v in views) == PATHS
    scene = st.Scene.from_scene(sc)
    g = torch.ones((sc.n_pixels, 3), device="cuda")

    def call():
        if adjoint:
            scene.backward(views, B, 1, g, st.make_opts(edge_term=0))
        else:
            scene.render(views, B, 1)
        s = scene.stats()
        assert s["device_error"] == 0
        return s["kernel_launches"]
    first, second = call(), call()
    scene.close()
    assert first - second in (0, 3)
    return first != second


@pytest.mark.parametrize("mesh,light,B,scale,adjoint,builds", [
    ("smooth", "env", 3, 1.0, True, True), ("smooth", "env", 1, 1.0, True, False), ("smooth", "view", 1, 1.0, True, True),
    ("smooth", "env", 3, 1.0, False, False),      # alone: 16.7 hits a face are not 19.5
    ("smooth", "env", 3, 30.0, True, False),      # edges over a unit long: the margins take too much
    ("fine fractal", "env", 3, 1.0, True, False), ("fine fractal", "view", 3, 1.0, True, False),
    ("knot", "env", 3, 1.0, True, True), ("knot", "env", 1, 1.0, True, False), ("knot", "env", 3, 1.0, False, False),
    ("knot", "view", 3, 1.0, True, True), ("knot", "view", 3, 1.0, False, False),
    ("small knot", "env", 3, 1.0, False, True), ("small knot", "env", 1, 1.0, True, True),
    ("rough", "env", 3, 1.0, True, False), ("rough", "view", 3, 1.0, True, False),
])
def test_rule(st, mesh, light, B, scale, adjoint, builds):  # noqa: F811
    assert _builds(st, mesh, light, B, scale, adjoint) == builds


def test_a_forward_call_counts_on_its_adjoint(st):  # noqa: F811
    """Alone it has too few paths; with an adjoint on the vertices before, whose build it shares, it builds them."""
    V, F = _mesh("smooth")
    rng = np.random.default_rng(2)
    views = S.fibonacci_views(4, [128] * 4, [128] * 4, [9] * 4)
    sc = S.Scene("rule", S._f32(V), np.ascontiguousarray(F, np.int32), S.random_face_params(rng, len(F)),
                 env=S.lognormal_env(rng, 64, 32), views=views, max_bounces=3)
    scene = st.Scene.from_scene(sc)
    W = torch.from_numpy(sc.vertices).cuda()

    def launches():
        scene.render(views, 3, 1)
        return scene.stats()["kernel_launches"]
    plain = launches()
    assert launches() == plain
    scene.backward(views, 3, 1, torch.ones((sc.n_pixels, 3), device="cuda"), st.make_opts(edge_term=0))
    used = launches()
    scene.refit(W)
    assert launches() == used + 3 and used == plain
    scene.close()


def test_paths_that_miss_do_not_count(st):  # noqa: F811
    """As many paths in wide views, most of which look past the mesh."""
    assert _builds(st, "smooth", "env", 3, 1.0, True)
    assert not _builds(st, "smooth", "env", 3, 1.0, True, w=512, h=32)


@pytest.mark.parametrize("side,light,n,adjoint,builds", [
    ("outer", "env", 48, True, True), ("outer", "env", 48, False, True), ("outer", "env", 64, False, False),
    ("outer", "env", 72, True, False), ("inner", "env", 8, True, False), ("inner", "view", 32, True, True),
    ("inner", "view", 80, True, False)])
def test_open_meshes(st, side, light, n, adjoint, builds):  # noqa: F811
    """Three planes of n x n quads each, 6 n^2 faces, from 2^21 paths on: the side that has directions is the one outward of
    the origin, where the planes see nothing (52 hits a face, alone 78) or one another (no build without traced lights)."""
    sc = S.color_bleed(n=n)
    rng = np.random.default_rng(2)
    views = S.fibonacci_views(4, [256] * 4, [256] * 4, [9] * 4)   # about 1.3 million hits
    if light == "view":
        views = S.with_view_lights(views)
    sc = S.Scene("open", S._f32(sc.vertices - (0.5 if side == "outer" else 0.0)), sc.faces, sc.face_params,
                 env=S.lognormal_env(rng, 64, 32) if light == "env" else None, views=views, max_bounces=3)
    assert sum(v.width * v.height * v.spp for v in views) >= 1 << 21
    scene = st.Scene.from_scene(sc)
    counts = []
    for _ in range(2):
        if adjoint:
            scene.backward(views, 3, 1, torch.ones((sc.n_pixels, 3), device="cuda"), st.make_opts(edge_term=0))
        else:
            scene.render(views, 3, 1)
        counts.append(scene.stats()["kernel_launches"])
        assert scene.stats()["device_error"] == 0
    scene.close()
    assert counts[0] - counts[1] == 6 + (3 if builds else 0)   # the primary lists, and the free directions
