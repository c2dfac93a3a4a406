"""Lists below 2048 references of quads on a few planes: the sort that spreads a depth's references by their
index, and its fallbacks (indices in clusters, two depths in one bucket)."""
import numpy as np
import pytest

from tests.scene_helpers import rects_scene
from tests.test_gpu_sort import _bin_lists, _check
from tests.test_gpu_sort_edges import lr  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [65, 66, 130, 257, 700, 1500, 2047])
@pytest.mark.parametrize("planes", [1, 2, 8, 30])
@pytest.mark.parametrize("kind", ["even", "clusters", "near", "mostly_one"])
def test_planes(lr, n, planes, kind):  # noqa: F811
    rng = np.random.default_rng(n * 31 + planes)
    z = 1.0 + np.arange(planes) / planes
    if kind == "near":                        # depths a few units in the last place apart: one bucket,
        z = 1.0 + np.arange(planes) * 2.0 ** -22
    depth = rng.choice(z, n)
    if kind == "mostly_one":
        depth = np.where(rng.random(n) < 0.9, 1.5, rng.uniform(1.0, 2.0, n))
    if kind == "near":
        depth[0] = 2.0                        # ... since another one is far away
    xy = np.floor(rng.uniform(0, 24, (n, 2)) * 4) / 4
    rects = [(float(x), float(y), float(x + 6.0), float(y + 5.0)) for x, y in xy]
    w = 32
    if kind == "clusters":                    # a second bin whose quads lie between the first one's two halves
        half, m = n // 2, 40 * n
        rects = rects[:half] + [(36.0, 2.0, 60.0, 20.0)] * m + rects[half:]
        depth = np.concatenate([depth[:half], rng.uniform(1.0, 2.0, m), depth[half:]])
        w = 64
    s = rects_scene(rects, width=w, height=32, depths=depth,
                    colors=np.concatenate([rng.random((len(rects), 3)), np.full((len(rects), 1), 0.1)], 1))
    st, bin_off, refs, rect = _bin_lists(lr, s)
    assert _check(s, st, bin_off, refs, rect)[0] == n
