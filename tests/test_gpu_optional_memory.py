"""Memory that a call can do without: screen records of edge candidates, wavefront engines past the second.

Where it is short, or would be large, the call runs with less of it and gives the same result.
"""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2012_03939_gb300 import scenes as S
from tests.test_gpu_bvh_builders import st  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


def _gradient(scene, sc, opts, B=2):
    w = torch.from_numpy(np.random.default_rng(1).normal(size=(sc.n_pixels, 3)).astype(np.float32)).cuda()
    g = torch.cat([x.ravel() for x in scene.backward(sc.views, B, 7, w, opts)]).cpu().numpy()
    assert scene.stats()["device_error"] == 0
    return g


def _close(got, ref):   # the scatter's FP32 atomics add in any order
    np.testing.assert_allclose(got, ref, rtol=1e-4, atol=1e-5 * np.abs(ref).max())


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _small():
    sc = S.tiny(res=40, spp=2)
    sc.views = S.ring_views(3, 40, 2)
    return sc


def test_edge_records_that_do_not_fit_are_done_without(st):  # noqa: F811
    sc, opts = _small(), st.make_opts(edge_term=1)
    scene = st.Scene.from_scene(sc)
    ref = _gradient(scene, sc, opts)
    scene.close()
    got = None
    for n in range(80):
        scene = st.Scene.from_scene(sc)
        st.inject_fault("alloc", n)
        try:
            got = _gradient(scene, sc, opts)
            break
        except st.StError as e:
            assert e.status == 2   # ST_ERR_OOM, of something the call needs
            scene.close()
    # the call went through although one of its allocations had failed: another one would fail now otherwise
    try:
        st.Scene.from_scene(sc).close()
    finally:
        st.inject_fault("alloc", -1)
    _close(got, ref)
    _close(_gradient(scene, sc, opts), ref)
    scene.close()


def test_edge_records_of_thousands_of_views_stay_small(st):  # noqa: F811
    V, F = S.uv_sphere(120, 62)   # 14640 faces, 21960 edges
    rng = np.random.default_rng(1)
    n = 3000
    sc = S.Scene("views", S._f32(V), np.ascontiguousarray(F, np.int32), S.random_face_params(rng, len(F)),
                 light_pos=S._f32([[3, 3, 3]]), light_intensity=S._f32([[5, 5, 5]]),
                 views=S.fibonacci_views(n, [8] * n, [8] * n, [1] * n), max_bounces=1)
    scene = st.Scene.from_scene(sc)
    _gradient(scene, dataclasses.replace(sc, views=sc.views[:1]), st.make_opts(edge_term=1), B=1)
    before = _free()
    got = _gradient(scene, sc, st.make_opts(edge_term=1), B=1)
    # 4 bytes of list an edge and view, and records within 256 MiB; 52 bytes an edge and view would be 3.4 GB
    assert before - _free() < 1 << 30
    # the same sum from calls of 500 views, whose records hold more candidates each
    ref = np.zeros_like(got, np.float64)
    other = st.Scene.from_scene(sc)
    w = torch.from_numpy(np.random.default_rng(1).normal(size=(sc.n_pixels, 3)).astype(np.float32)).cuda()
    for a in range(0, n, 500):
        ref += torch.cat([x.ravel() for x in other.backward(sc.views[a:a + 500], 1, 7, w, st.make_opts(edge_term=1))]).double().cpu().numpy()
    _close(got, ref)
    scene.close()
    other.close()


def _chunked(st, **kw):
    return st.make_opts(chunk_paths=2048, **kw)   # 9600 paths: five chunks, so four engines where they fit


def _image(scene, sc, opts):
    img = scene.render(sc.views, 2, 7, opts).cpu().numpy()
    assert scene.stats()["device_error"] == 0
    return img


def test_further_engines_that_do_not_fit_are_done_without(st):  # noqa: F811
    sc = _small()
    scene = st.Scene.from_scene(sc)
    ref = _image(scene, sc, _chunked(st))
    full = scene.stats()["scratch_bytes"]
    scene.close()
    held = []
    for n in range(120):
        scene = st.Scene.from_scene(sc)
        with pytest.raises(st.StError):
            scene.render([], 2, 7, out=torch.zeros((sc.n_pixels, 3), device="cuda"))
        said = st.lib().st_last_error()
        st.inject_fault("alloc", n)
        try:
            img = _image(scene, sc, _chunked(st))
        except st.StError as e:
            assert e.status == 2
            st.inject_fault("alloc", -1)
            np.testing.assert_array_equal(_image(scene, sc, _chunked(st)), ref)
            scene.close()
            continue
        finally:
            st.inject_fault("alloc", -1)
        np.testing.assert_array_equal(img, ref)
        assert st.lib().st_last_error() == said   # nothing was refused
        held.append(scene.stats()["scratch_bytes"])
        np.testing.assert_array_equal(_image(scene, sc, _chunked(st)), ref)
        scene.close()
        if held[-1] == full:
            break
    # first without the third and the fourth engine, then without the fourth, then with all of them
    assert sorted(set(held)) == [full // 2, full // 4 * 3, full]


@pytest.mark.parametrize("backward", [False, True])
def test_further_engines_are_given_back_where_memory_is_short(st, backward):  # noqa: F811
    """A later call's buffers do not fit beside the optional engines: they go, and the call succeeds."""
    sc, big = _small(), S.tiny(res=72, spp=3)
    big.views = S.ring_views(5, 72, 3)
    call = _gradient if backward else _image
    opts = _chunked(st, edge_term=1 if backward else 0)
    fresh = st.Scene.from_scene(big)
    ref = call(fresh, big, opts)
    fresh.close()
    for n in range(200):
        scene = st.Scene.from_scene(sc)
        call(scene, sc, opts)
        before = scene.stats()["scratch_bytes"]
        st.inject_fault("alloc", n)
        try:
            got = call(scene, big, opts)   # no allocation's failure reaches the caller while engines can be given back
        finally:
            st.inject_fault("alloc", -1)
        (_close if backward else np.testing.assert_array_equal)(got, ref)
        after = scene.stats()["scratch_bytes"]
        (_close if backward else np.testing.assert_array_equal)(call(scene, big, opts), ref)
        scene.close()
        if n == 0:
            assert after < before   # the tables came first: two engines stayed
        st.inject_fault("alloc", -1)
        if n > 6:
            return
