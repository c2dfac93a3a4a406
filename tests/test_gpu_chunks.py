"""Binning chunks: quad counts around the chunk sizes, and large quads around the number of bins
from which the whole CTA shares one (more than 128 bins: 11x12 bins are above, 8x16 are not)."""
import numpy as np
import pytest
import torch

import oracle
import scenegen
from tests.test_gpu_raster_batches import check, rgba, scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lr():
    import paper_2405_13364_gb300 as P
    P.load_library()
    return P


@pytest.mark.parametrize("n", [1, 255, 256, 257, 511, 513, 1025, 2049])
@pytest.mark.parametrize("box", [(256, 512), (352, 384), (600, 600)])
def test_large_quads(lr, n, box):
    rng = np.random.default_rng(n + box[0])
    w, h, m = 523, 517, min(n, 40)
    xy = rng.uniform(0, [w, h], (n, 1, 2)) + rng.uniform(0, 6, (n, 4, 2))
    # m of them span up to box px: random (convex, concave, crossed), and exact rectangles
    big = rng.choice(n, m, replace=False)
    o = rng.uniform(-100, [w - box[0] + 100, h - box[1] + 100], (m, 1, 2))
    xy[big] = o + rng.uniform(0, 1, (m, 4, 2)) * box
    rect = np.array([[0, 0], [1, 0], [1, 1], [0, 1]]) * np.array(box)
    xy[big[::3]] = np.floor(o[::3] / 32) * 32 + rect
    z = np.where(rng.random((n, 1)) < 0.5, 1.0, rng.uniform(1.0, 2.0, (n, 4)))
    check(lr, scene(xy, z, rgba(rng, n), w, h), 3)


def test_chunks_of_a_batch(lr):
    # views of very different size share one chunk size; every view equals its own render
    sizes = [(3, 64, 64), (700, 333, 190), (5000, 640, 360)]
    scenes = [scenegen.frustum_parallelograms(q, w, h, seed=q) for q, w, h in sizes]
    r = lr.Renderer(sorter_k=3)
    outs = r.render_batch([(lr.DeviceScene.from_scene(s), s.width, s.height) for s in scenes], count=True)
    torch.cuda.synchronize()
    for s, o in zip(scenes, outs):
        assert np.array_equal(o["count"].cpu().numpy().view(np.uint32), oracle.render(s)["count"])
    r.close()
