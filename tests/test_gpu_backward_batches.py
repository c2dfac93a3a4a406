"""The backward's per-batch sums: stacks in which every pixel has more fragments of a batch than
are recorded, batch remainders, nearly opaque and nearly transparent quads, against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from tests.test_gpu_raster_batches import rgba, scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 3, 12])
@pytest.mark.parametrize("n", [1, 12, 13, 31, 32, 33, 65, 200])
@pytest.mark.parametrize("full", [True, False])
def test_stack(k, n, full):
    import paper_2405_13364_gb300 as P
    rng = np.random.default_rng(n + 7 * full)
    w, h = 21, 13
    if full:                                   # every quad covers every pixel
        xy = np.tile(np.array([[-1.0, -1.0], [w + 1, -1], [w + 1, h + 1], [-1, h + 1]]), (n, 1, 1))
    else:
        xy = rng.uniform(-4, [w, h], (n, 1, 2)) + rng.uniform(0, 12, (n, 4, 2))
    z = rng.uniform(1.0, 2.0, (n, 1)) + rng.uniform(0, 0.05, (n, 4)) * (rng.random((n, 1)) < 0.7)
    col = rgba(rng, n, 0.02, 0.4).astype(np.float32)
    col[::17, 3] = 0.9
    col[5::17, 3] = 1e-4
    s = scene(xy, z, col, w, h)
    r = P.Renderer(sorter_k=k)
    colors = torch.tensor(col, device="cuda", requires_grad=True)
    img = P.composite(colors, r, P.DeviceScene.from_scene(s), w, h)
    g_out = rng.standard_normal((h, w, 4)).astype(np.float32)
    img.backward(torch.tensor(g_out, device="cuda"))
    g = colors.grad.cpu().numpy().astype(np.float64)
    ref = oracle.backward(s, g_out.astype(np.float64), col.astype(np.float64))
    # the backward suite's 1e-3, and for quads far behind, whose gradient is a difference of sums in
    # fp32, the colour tolerance of 1e-5 relative to the largest gradient
    assert np.all(np.abs(g - ref) <= 1e-3 * np.abs(ref) + 1e-5 * np.abs(ref).max())
    r.close()
