"""An infinite loss gradient at one pixel stays infinite, and not a NaN, in the gradient of the opaque quad
in front, whose alpha gradient has no term of what lies behind it."""
import numpy as np
import pytest
import torch

from tests.test_gpu_raster_batches import rgba, scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 3, 8])
@pytest.mark.parametrize("behind", [0, 1, 40])
def test_opaque_front(k, behind):
    import paper_2405_13364_gb300 as P
    rng = np.random.default_rng(behind)
    n, w, h = behind + 1, 21, 13
    xy = np.tile(np.array([[-1.0, -1.0], [w + 1, -1], [w + 1, h + 1], [-1, h + 1]]), (n, 1, 1))
    col = rgba(rng, n, 0.1, 0.4).astype(np.float32)
    col[0] = (0.5, 0.25, 0.75, 1.0)
    r = P.Renderer(sorter_k=k)
    colors = torch.tensor(col, device="cuda", requires_grad=True)
    img = P.composite(colors, r, P.DeviceScene.from_scene(scene(xy, np.linspace(1.0, 2.0, n)[:, None], col, w, h)), w, h)
    g_out = np.zeros((h, w, 4), np.float32)
    g_out[5, 7, 0] = np.inf
    img.backward(torch.tensor(g_out, device="cuda"))
    g = colors.grad[0].cpu().numpy()
    assert np.array_equal(g, np.array([np.inf, 0.0, 0.0, np.inf], np.float32)), g
    r.close()
