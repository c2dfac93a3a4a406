"""Bins whose sorted list is every pixel's exact order have a rasteriser of their own. Its image is, bit
for bit, that of the per-pixel sorter (which takes every bin when the coverage hash is asked for),
whatever else is in the batch, whatever other outputs are asked for, however long the lists are and
however a bin is divided over warps; and what the backward recomputes is that image's own sums."""
import numpy as np
import pytest
import torch

import oracle
import scenegen
from paper_2405_13364_gb300 import partition as PT
from tests.test_gpu_boxes import boxes
from tests.test_gpu_raster_batches import rgba, scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lr():
    import paper_2405_13364_gb300 as P
    P.load_library()
    return P


def sprites(n, w, h, shape, seed):
    """Quads of constant depth: upright rectangles, other quads (concave and crossed ones too), or both."""
    rng = np.random.default_rng(seed)
    xy = boxes(rng, n, w, h, 0.2, 20.0)
    z = np.round(rng.uniform(1.0, 2.0, (n, 1)), 3)                       # some depths equal
    if shape != "rects":
        odd = slice(None) if shape == "others" else rng.choice(n, 3, replace=False)
        xy[odd] = xy[odd, :1] + rng.uniform(0, 15, xy[odd].shape)
    return scene(xy, z, rgba(rng, n, 0.02, 0.2), w, h)


@pytest.mark.parametrize("shape", ["rects", "others", "both"])
@pytest.mark.parametrize("bin_size", [16, 32, 64])
@pytest.mark.parametrize("size", [(5, 3), (33, 21), (70, 67), (129, 100)])
@pytest.mark.parametrize("n", [300, 9000])
def test_equals_per_pixel_sorter(lr, shape, bin_size, size, n):
    w, h = size
    s = lr.DeviceScene.from_scene(sprites(n, w, h, shape, n + w + bin_size))
    r = lr.Renderer(sorter_k=1, bin_size=bin_size)
    ref = r.render(s, w, h, rgba8=True, count=True, hash=True)
    for opts in ({}, {"rgba8": True}, {"count": True, "exact_mask": True}):
        out = r.render(s, w, h, **opts)
        for name in opts if "exact_mask" not in opts else ["count"]:
            assert torch.equal(out[name], ref[name])
        assert torch.equal(out["rgba"], ref["rgba"])
        if "exact_mask" in opts:
            assert not out["exact_mask"].any()
    # a tile per rank: its pixels as in the whole image, the others untouched
    owner = PT.assign_tiles(w, h, 2)
    for rank in range(2):
        bits = torch.from_numpy(PT.owned_bitset(owner, rank).view(np.int32)).cuda()
        out = r.make_outputs(w, h)
        out["rgba"].fill_(-1.0)
        r.render(s, w, h, owned_tiles=bits, out=out)
        mine = torch.zeros((h, w), dtype=torch.bool, device="cuda")
        for x0, y0, x1, y1 in PT.tile_rects(owner, rank, w, h):
            mine[y0:y1, x0:x1] = True
        assert torch.equal(out["rgba"], torch.where(mine[..., None], ref["rgba"], torch.full_like(ref["rgba"], -1.0)))
    r.close()


def test_alone_in_a_batch_and_served(lr):
    # 470,000 references in lists of up to 8000, beside a view with 2.5M of them
    w, h = 640, 360
    small = lr.DeviceScene.from_scene(scenegen.gaussian_particles(300_000, w, h, seed=1))
    large = lr.DeviceScene.from_scene(scenegen.gaussian_particles(1_600_000, 1920, 1080, seed=2))
    r = lr.Renderer(sorter_k=3)
    alone = r.render(small, w, h)["rgba"]
    assert torch.equal(r.render(small, w, h, rgba8=True)["rgba"], alone)
    assert torch.equal(r.render(small, w, h, hash=True)["rgba"], alone)
    assert torch.equal(r.render_batch([(small, w, h), (large, 1920, 1080)])[0]["rgba"], alone)
    assert torch.equal(r.render_batch([(large, 1920, 1080)] * 2 + [(small, w, h)])[2]["rgba"], alone)
    r.close()
    srv = lr.Server(sorter_k=3, num_slots=1, max_batch_views=4, slot_workspace_bytes=2 << 30)
    tickets = [srv.submit(s, *size) for s, size in [(large, (1920, 1080))] + [(small, (w, h)), (large, (1920, 1080))] * 2]
    done = [srv.poll(t, timeout_us=10_000_000) for t in tickets]
    torch.cuda.synchronize()
    assert all(d is not None and d[0] == 0 for d in done)
    assert any(d[2]["batch_views"] > 1 for d in done)
    for d in (done[1], done[3]):
        assert torch.equal(d[1]["rgba"], alone)
    srv.close()


def test_gradient_of_a_nearly_opaque_quad_behind_a_long_list(lr):
    # behind the deepest quad lies nothing, so that its alpha gradient is T g . c whatever 1 / (1 - a) is
    n, w, h = 1500, 32, 32
    rng = np.random.default_rng(3)
    xy = np.tile(np.array([[-2.0, -2.0], [w + 2, -2], [w + 2, h + 2], [-2, h + 2]]), (n, 1, 1))
    col = rgba(rng, n, 0.0005, 0.002).astype(np.float32)
    col[-1, 3] = 1.0 - 1e-5
    s = scene(xy, np.linspace(1.0, 2.0, n)[:, None], col, w, h)
    r = lr.Renderer(sorter_k=3)
    colors = torch.tensor(col, device="cuda", requires_grad=True)
    img = lr.composite(colors, r, lr.DeviceScene.from_scene(s), w, h)
    g_out = rng.standard_normal((h, w, 4)).astype(np.float32)
    g_out[..., 3] = 0.0                        # (the image holds 1 - T, so T itself is not known that well)
    img.backward(torch.tensor(g_out, device="cuda"))
    g = colors.grad.cpu().numpy().astype(np.float64)
    ref = oracle.backward(s, g_out.astype(np.float64), col.astype(np.float64))
    # the bound of the backward's other stacks
    assert np.all(np.abs(g - ref) <= 1e-3 * np.abs(ref) + 1e-5 * np.abs(ref).max())
    r.close()
