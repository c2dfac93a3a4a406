"""The per-quad words that lr_ws_layout describes: rec_info bit by bit from the snapped vertices, and the
record's info word, which is the same for a visible quad."""
import numpy as np
import pytest
import torch

from paper_2405_13364_gb300 import _binding as B
from tests.test_gpu_boxes import boxes
from tests.test_gpu_raster_batches import rgba, scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("outputs", [{}, {"hash": True}])
def test_info_words(outputs):
    import paper_2405_13364_gb300 as P
    rng = np.random.default_rng(2)
    w, h, n = 700, 500, 1200
    xy = boxes(rng, n, w, h, 0.2, 20.0)                                       # upright rectangles
    xy[::3] = xy[::3, :1] + rng.uniform(0, 30, xy[::3].shape)                 # other quads
    xy[1::5] = boxes(rng, len(xy[1::5]), w, h, 100.0, 400.0)                  # large rectangles
    xy[2::50, 2] = xy[2::50, 0]                                               # a triangle without area
    z = np.where(np.arange(n)[:, None] % 2 == 0, 1.5, rng.uniform(1.0, 2.0, (n, 4)))
    s = scene(xy, z, rgba(rng, n), w, h)
    ds = P.DeviceScene.from_scene(s)
    r = P.Renderer()
    out = r.make_outputs(w, h, **outputs)
    view = r.view_struct(ds, w, h, out)
    r.render_views([view])
    torch.cuda.synchronize()
    lay = B.lr_workspace_layout(r.ctx, [view], r._ws_bytes)
    off = -int(r._ws.data_ptr()) % 256

    def grab(at, words):
        return r._ws[off + at: off + at + 4 * words].cpu().numpy().view(np.uint32)

    rec, info = grab(lay.rec, 16 * n).reshape(n, 16), grab(lay.rec_info, n)
    r.close()
    vis = (info >> 8) == 0
    assert vis.sum() > 900
    rec, info = rec[vis], info[vis]
    assert np.array_equal(rec[:, 14], info)
    X, Y = rec[:, 0:8:2].view(np.int32).astype(np.int64), rec[:, 1:8:2].view(np.int32).astype(np.int64)
    q = rec[:, 8:12].view(np.float32)
    area = [(X[:, b] - X[:, 0]) * (Y[:, c] - Y[:, 0]) - (Y[:, b] - Y[:, 0]) * (X[:, c] - X[:, 0]) for b, c in ((1, 2), (2, 3))]
    for t in range(2):
        assert np.array_equal(info >> t & 1, area[t] != 0)
        assert np.array_equal(info >> (4 + t) & 1, area[t] < 0)
        # 32-bit edge values wherever a half-block touches the triangle's box: 7 px to its sides, 3 above and below
        tri = [0, 1 + t, 2 + t]
        wx, wy = np.ptp(X[:, tri], axis=1), np.ptp(Y[:, tri], axis=1)
        small = (wx < 32768) & (wy < 32768) & (wx * (wy + 768) + wy * (wx + 1792) + 1 < 1 << 30)
        assert 0 < small.sum() < len(small)
        assert np.array_equal(info >> (6 + t) & 1, small & (area[t] != 0))
    assert np.array_equal(info >> 3 & 1, (q == q[:, :1]).all(1))
    boxed = ((X[:, 0] == X[:, 3]) & (X[:, 1] == X[:, 2]) & (Y[:, 0] == Y[:, 1]) & (Y[:, 2] == Y[:, 3])) | \
            ((X[:, 0] == X[:, 1]) & (X[:, 2] == X[:, 3]) & (Y[:, 0] == Y[:, 3]) & (Y[:, 1] == Y[:, 2]))
    assert boxed.any() and np.array_equal(rec[:, 15] >> 1 & 1, boxed)
