"""The lists' two passes agree: as many leaves are written to a cell as were counted for it.

Each pass projects the leaves for itself. On a mesh of a million faces some corners fall on a cell's padded border within
rounding, and a leaf that only one of the passes takes there leaves a cell's list one too short (a leaf is dropped, whichever
comes last) or with an entry that was never written. Either sets the device error.
"""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2012_03939_gb300 import scenes as S
from tests.test_gpu_bvh_builders import st  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("jitter", [0.0, 0.0005])
def test_every_counted_leaf_is_written(st, jitter):  # noqa: F811
    sc = S.make("scale")
    scene = st.Scene.from_scene(sc)
    if jitter:
        V = sc.vertices + np.random.default_rng(1).normal(0, jitter, sc.vertices.shape)
        scene.refit(torch.from_numpy(S._f32(V)).cuda())
    for first in range(0, len(sc.views), 8):
        views, off = [], 0
        for v in sc.views[first:first + 8]:
            views.append(dataclasses.replace(v, spp=1, pixel_offset=off))
            off += v.width * v.height
        assert off >= 1 << 20   # primary and light lists
        scene.render(views, 1, 1)
        assert scene.stats()["device_error"] == 0, first
    scene.close()
