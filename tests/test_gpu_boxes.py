"""Bins that hold axis-parallel rectangles of constant depth only, rasterised in 16x8 blocks:
image sizes that cut the blocks everywhere, edges through and between pixel centres, every bin
size, windows of more than 1024 references, and bins that also hold one quad of another kind."""
import numpy as np
import pytest
import torch

import oracle
from tests.test_gpu_raster_batches import check, rgba, scene
from tests.test_gpu_threshold import assert_threshold_parity, render_threshold

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lr():
    import paper_2405_13364_gb300 as P
    P.load_library()
    return P


def boxes(rng, n, w, h, lo, hi, grid=1):
    o = rng.uniform(-hi, [w, h], (n, 1, 2))
    wh = rng.uniform(lo, hi, (n, 1, 2))
    wh = np.where(rng.random((n, 1, 1)) < 0.5, wh, np.round(wh))
    xy = o + wh * np.array([[0, 0], [1, 0], [1, 1], [0, 1]])
    xy = np.round(xy * 256 / grid) * grid / 256
    k = rng.integers(0, 4, n)                       # any corner first, either winding
    xy = np.stack([np.roll(q, -s, 0) for q, s in zip(xy, k)])
    flip = rng.random(n) < 0.5
    xy[flip] = xy[flip, ::-1]
    return xy


@pytest.mark.parametrize("size", [(1, 1), (7, 3), (8, 4), (9, 5), (15, 8), (16, 9), (17, 7), (31, 33), (47, 40), (203, 141)])
@pytest.mark.parametrize("grid", [1, 128])
@pytest.mark.parametrize("bin_size", [16, 32, 64])
def test_boxes(lr, size, grid, bin_size):
    rng = np.random.default_rng(size[0] * 1000 + size[1] + grid + bin_size)
    w, h = size
    n = 1500 if w < 100 else 4000
    xy = boxes(rng, n, w, h, 0.2, 20.0, grid)
    s = scene(xy, rng.uniform(1.0, 2.0, (n, 1)), rgba(rng, n, 0.02, 0.2), w, h)
    check(lr, s, 1, bin_size=bin_size)
    s = scene(xy, np.round(rng.uniform(1.0, 2.0, (n, 1)) * 4) / 4, rgba(rng, n, 0.02, 0.2), w, h)   # equal depths
    check(lr, s, 3, bin_size=bin_size)


@pytest.mark.parametrize("other", ["rotated", "tilted"])
def test_boxes_among_other_quads(lr, other):
    rng = np.random.default_rng(5)
    w, h, n = 203, 141, 3000
    xy = boxes(rng, n, w, h, 1.0, 12.0)
    z = np.repeat(rng.uniform(1.0, 2.0, (n, 1)), 4, 1)
    odd = rng.choice(n, 12, replace=False)
    if other == "rotated":
        xy[odd] = rng.uniform(0, [w, h], (12, 1, 2)) + np.array([[0, -9], [9, 0], [0, 9], [-9, 0]])
    else:
        z[odd, 1:3] += 0.1
    check(lr, scene(xy, z, rgba(rng, n, 0.02, 0.2), w, h), 1)


def test_boxes_threshold(lr):
    rng = np.random.default_rng(6)
    w, h, n = 203, 141, 6000
    s = scene(boxes(rng, n, w, h, 2.0, 20.0), rng.uniform(1.0, 2.0, (n, 1)), rgba(rng, n, 0.1, 0.4), w, h)
    g, _ = render_threshold(lr, s, 1)
    assert_threshold_parity(g, s)


@pytest.mark.parametrize("n", [1000, 1023, 1024, 1025, 2300, 4097, 20000, 66000])
@pytest.mark.parametrize("bin_size", [16, 32, 64])
def test_long_lists(lr, n, bin_size):
    # lists composited by a CTA's warps in segments (one bin of every size holds all), with and without
    # counts
    rng = np.random.default_rng(n)
    w = h = 16
    xy = rng.uniform(0, w - 4, (n, 1, 2)) + rng.uniform(1.0, 4.0, (n, 1, 2)) * np.array([[0, 0], [1, 0], [1, 1], [0, 1]])
    s = scene(xy, rng.uniform(1.0, 2.0, (n, 1)), rgba(rng, n, 0.0005, 0.003), w, h)
    ref = oracle.render(s)
    r = lr.Renderer(sorter_k=1, bin_size=bin_size)
    d = lr.DeviceScene.from_scene(s)
    for count in (False, True, False):
        out = r.render(d, w, h, count=count, exact_mask=True)
        torch.cuda.synchronize()
        assert np.abs(out["rgba"].cpu().numpy().astype(np.float64) - ref["rgba"]).max() <= 1e-5
        assert not out["exact_mask"].any()
        if count:
            assert np.array_equal(out["count"].cpu().numpy().view(np.uint32), ref["count"])
        assert r.stats()["fragments"] == int(ref["count"].astype(np.int64).sum())
    r.close()


@pytest.mark.parametrize("n", [1023, 1024, 5000])
@pytest.mark.parametrize("bin_size", [16, 32, 64])
def test_long_lists_of_other_shapes(lr, n, bin_size):
    # constant depths, not all axis-parallel: eight 8x8 blocks at a time
    rng = np.random.default_rng(n + bin_size)
    w, h = 75, 67
    xy = rng.uniform(0, [w, h], (n, 1, 2)) + rng.uniform(2.0, 9.0, (n, 1, 1)) * np.array([[0, -1], [1, 0], [0, 1], [-1, 0]])
    xy[: n // 2] = rng.uniform(0, 30, (n // 2, 1, 2)) + rng.uniform(2.0, 30.0, (n // 2, 1, 2)) * np.array([[0, 0], [1, 0], [1, 1], [0, 1]])
    check(lr, scene(xy, rng.uniform(1.0, 2.0, (n, 1)), rgba(rng, n, 0.01, 0.05), w, h), 1, bin_size=bin_size)


@pytest.mark.parametrize("n", [900, 3000, 30000])
@pytest.mark.parametrize("bin_size", [16, 32, 64])
def test_long_lists_bytes(lr, n, bin_size):
    # 8-bit values are those of the list blended in one go, as the hashing rasteriser blends it
    rng = np.random.default_rng(n)
    w, h = 75, 67
    xy = boxes(rng, n, w, h, 1.0, 30.0)
    s = scene(xy, rng.uniform(1.0, 2.0, (n, 1)), rgba(rng, n, 0.005, 0.05), w, h)
    r = lr.Renderer(sorter_k=1, bin_size=bin_size)
    d = lr.DeviceScene.from_scene(s)
    a = r.render(d, w, h, rgba8=True, count=True)
    b = r.render(d, w, h, rgba8=True, count=True, hash=True)
    assert torch.equal(a["rgba8"], b["rgba8"]) and torch.equal(a["count"], b["count"])
    assert torch.equal(a["rgba"], b["rgba"])
    r.close()
