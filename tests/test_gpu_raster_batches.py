"""The rasteriser's batches against the oracle, on the kernel instances without the coverage
hash: the fp32 interval masks at the limits of their range (edges up to 128 px, subpixel
positions and edges through pixel centres), the integer masks above it, quads of constant
depth blended in stream order, and half-blocks that change between the two."""
import numpy as np
import pytest
import torch

import oracle
import scenegen
from scenegen import COLOR_FLAT, COLOR_VERTEX, Scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lr():
    import paper_2405_13364_gb300 as P
    P.load_library()
    return P


def scene(xy, z, colors, w, h, mode=COLOR_FLAT):
    """Quads at screen positions xy [Q][4][2] and view depths z [Q][4]."""
    m, n, f = scenegen.pixel_pinhole(w, h)
    z = np.broadcast_to(np.asarray(z, np.float64), xy.shape[:2])
    pos = np.concatenate([xy * z[..., None], z[..., None]], -1).reshape(-1, 3).astype(np.float32)
    return Scene(pos, None, np.asarray(colors, np.float32), mode, m, float(n), float(f), w, h)


def rgba(rng, n, lo=0.1, hi=0.6):
    return np.concatenate([rng.random((n, 3)), rng.uniform(lo, hi, (n, 1))], 1)


def check(lr, s, k, **opts):
    ref = oracle.render(s)
    r = lr.Renderer(sorter_k=k, **opts)
    out = r.render(lr.DeviceScene.from_scene(s), s.width, s.height, count=True)
    torch.cuda.synchronize()
    got, cnt = out["rgba"].cpu().numpy().astype(np.float64), out["count"].cpu().numpy().view(np.uint32)
    r.close()
    assert np.array_equal(cnt, ref["count"])
    assert np.abs(got - ref["rgba"]).max() <= 1e-5      # the parity suite's colour tolerance
    return ref


@pytest.mark.parametrize("side", [0.6, 8.0, 127.5, 127.996, 128.0, 128.5, 400.0])
@pytest.mark.parametrize("grid", [1, 128, 256])       # vertex positions in 1/256 px multiples
def test_masks(lr, side, grid):
    # random quads (convex, concave, crossed, both windings) whose box is up to `side` px, on
    # positions that put edges off, through and between pixel centres
    rng = np.random.default_rng(int(side * 1000) + grid)
    n, w, h = 600, 203, 141
    xy = rng.uniform(-side / 2, [w, h], (n, 1, 2)) + rng.uniform(0, side, (n, 4, 2))
    xy = np.round(xy * 256 / grid) * grid / 256
    xy[::5, 1, 1] = xy[::5, 0, 1]                     # horizontal and vertical edges
    xy[1::5, 2, 0] = xy[1::5, 1, 0]
    z = np.where(rng.random((n, 1)) < 0.5, 1.0, rng.uniform(1.0, 2.0, (n, 4)))
    check(lr, scene(xy, z, rgba(rng, n), w, h), 3)
    check(lr, scene(xy, z, rgba(rng, 4 * n), w, h, COLOR_VERTEX), 1)


@pytest.mark.parametrize("k", [1, 2, 3, 8])
@pytest.mark.parametrize("opts", [{}, {"carry_colors": True}, {"bin_size": 64}])
@pytest.mark.parametrize("tilted", [0.0, 0.02, 0.5])  # share of quads not of constant depth
def test_constant_depths(lr, k, opts, tilted):
    # more than a batch per half-block, equal depths, quads whose triangles overlap
    rng = np.random.default_rng(k + int(100 * tilted))
    n, w, h = 3000, 61, 43
    xy = rng.uniform(-6, [w, h], (n, 1, 2)) + rng.uniform(0, 12, (n, 4, 2))
    sq = np.array([[0, 0], [1, 0], [1, 1], [0, 1]])
    boxes = rng.random(n) < 0.7
    xy[boxes] = xy[boxes, :1] + sq * rng.uniform(1, 12, (int(boxes.sum()), 1, 1))
    z = np.round(rng.uniform(1.0, 3.0, (n, 1)) * 64) / 64 * np.ones((1, 4))
    t = rng.random(n) < tilted
    z[t] += rng.uniform(0, 0.3, (int(t.sum()), 4))
    ref = check(lr, scene(xy, z, rgba(rng, n), w, h), k, **opts)
    assert ref["count"].max() > 32     # more than one batch at a pixel


@pytest.mark.parametrize("k", [1, 3])
def test_constant_depths_threshold(lr, k):
    rng = np.random.default_rng(k)
    n, w, h = 4000, 61, 43
    sq = np.array([[0, 0], [1, 0], [1, 1], [0, 1]])
    xy = rng.uniform(-6, [w, h], (n, 1, 2)) + sq * rng.uniform(1, 14, (n, 1, 1))
    z = rng.uniform(1.0, 3.0, (n, 1)) * np.ones((1, 4))
    z[::40] += rng.uniform(0, 0.3, (z[::40].shape[0], 4))
    s = scene(xy, z, rgba(rng, n), w, h)
    ref = oracle.render_threshold(s, 1.0 / 128.0)
    r = lr.Renderer(sorter_k=k, alpha_threshold=True)
    got = r.render(lr.DeviceScene.from_scene(s), w, h)["rgba"].cpu().numpy().astype(np.float64)
    r.close()
    assert np.abs(got - ref["rgba"]).max() <= 1e-5


@pytest.mark.parametrize("size,bin_size", [((2560, 2048), 16), ((2560, 2048), 32), ((9, 5), 32)])
def test_constant_depths_sizes(lr, size, bin_size):
    # more bins than the binning CTAs count in shared memory, two half-blocks per ticket, a
    # frame smaller than a bin; no pixel takes the exact path
    w, h = size
    s = scenegen.gaussian_particles(30_000 if w > 9 else 300, w, h, seed=bin_size)
    ref = oracle.render(s)
    r = lr.Renderer(sorter_k=3, bin_size=bin_size)
    out = r.render(lr.DeviceScene.from_scene(s), w, h, count=True, exact_mask=True)
    torch.cuda.synchronize()
    assert np.array_equal(out["count"].cpu().numpy().view(np.uint32), ref["count"])
    assert np.abs(out["rgba"].cpu().numpy().astype(np.float64) - ref["rgba"]).max() <= 1e-5
    assert not out["exact_mask"].any()
    assert r.stats()["fragments"] == int(ref["count"].sum())
    r.close()
