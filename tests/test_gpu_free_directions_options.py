"""Free directions under every shading option and light, in the images and in the gradients.

One call that uses them against its views each in a call too small to: both shading kernels take the same decisions and
add the same terms, so images, signatures and ray counts are equal bitwise; the gradients differ by the order in which FP32
atomics add.
"""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2012_03939_gb300 import scenes as S
from tests.test_gpu_bvh_builders import st  # noqa: F401  (the fixture)
from tests.test_gpu_free_directions_meshes import _equal_to_small_calls

pytestmark = pytest.mark.gpu

OPTIONS = [  # brdf, fresnel, RGB specular, color_res, smooth
    ("ggx", 0, False, 0, False), ("ggx", 1, True, 2, True), ("ggx", 0, False, 1, True), ("beckmann", 0, False, 0, False),
    ("beckmann", 0, False, 3, True), ("beckmann", 1, True, 0, True), ("beckmann", 1, False, 2, False)]
LIGHTS = ["env", "points", "view", "all"]


def _scene(opt, light, seed):
    brdf, fresnel, rgb, res, smooth = opt
    rng = np.random.default_rng(seed)
    V, F = S.uv_sphere(60, 31)
    V = S.fractal_displace(V, rng, amp=0.12)
    P = S.random_face_params(rng, len(F) * (res + 1) * (res + 2) // 2)
    if rgb:
        P = np.concatenate([P[:, :3], rng.uniform(0.02, 0.3, size=(len(P), 3)).astype(np.float32), P[:, 4:]], 1)
    lp = S._f32([[2.0, 1.5, 2.5], [-0.3, 3.0, 0.2]] if light in ("points", "all") else np.zeros((0, 3)))
    views = S.fibonacci_views(2, [131, 128], [128, 111], [16, 20])
    if light in ("view", "all"):
        views = S.with_view_lights(views)
    return S.Scene("options", S._f32(V), np.ascontiguousarray(F, np.int32), P, brdf, light_pos=lp,
                   light_intensity=np.full_like(lp, 5.0), env=S.lognormal_env(rng, 64, 32) if light in ("env", "all") else None,
                   views=views, max_bounces=4, color_res=res, smooth_normals=smooth, fresnel=fresnel)


@pytest.mark.parametrize("light", LIGHTS)
@pytest.mark.parametrize("opt", OPTIONS)
def test_images_under_every_option(st, opt, light):  # noqa: F811
    sc = _scene(opt, light, 5)
    scene = st.Scene.from_scene(sc)
    for seed in (5, 6, 7):
        many, few = _equal_to_small_calls(st, scene, sc, seed=seed)
    assert many["node_visits"] < 0.97 * few["node_visits"]   # they answered bounce rays (most fetches are first rays')
    scene.close()


@pytest.mark.parametrize("term", [0, 1, 3, 5])
@pytest.mark.parametrize("opt,light", [(OPTIONS[0], "env"), (OPTIONS[1], "all"), (OPTIONS[4], "view"), (OPTIONS[5], "points"),
                                       (OPTIONS[6], "all")])
def test_gradients_under_every_term(st, opt, light, term):  # noqa: F811
    if term == 5 and light == "env":
        pytest.skip("shadow edges need a point light")
    sc = _scene(opt, light, 6)
    scene = st.Scene.from_scene(sc)
    w = torch.from_numpy(np.random.default_rng(2).normal(size=(sc.n_pixels, 3)).astype(np.float32)).cuda()
    o = st.make_opts(edge_term=term, edge_spp=1, count_visits=1)
    counts = ("extension_rays", "shadow_rays", "secondary_samples", "edge_samples")
    dV, dF = scene.backward(sc.views, 4, 9, w, o)
    many = scene.stats()
    rV, rF, few, visits = torch.zeros_like(dV, dtype=torch.float64), torch.zeros_like(dF, dtype=torch.float64), dict.fromkeys(counts, 0), 0
    for v in sc.views:
        a, b = scene.backward([v], 4, 9, w, o)
        rV += a
        rF += b
        s = scene.stats()
        assert s["device_error"] == 0
        visits += s["node_visits"]
        for k in counts:
            few[k] += s[k]
    assert many["device_error"] == 0 and {k: many[k] for k in counts} == few
    assert many["node_visits"] < visits
    for got, ref in ((dV, rV), (dF, rF)):
        got, ref = got.double().cpu().numpy(), ref.cpu().numpy()
        np.testing.assert_allclose(got, ref, rtol=1e-4, atol=1e-5 * np.abs(ref).max())
    scene.close()
