"""The per-bin depth sort at the sizes where its form changes: the quarter-CTA bucket sort's
keys per thread (256, 512, 768 and 1024 references), the high-density limit (2048), the bucket
sort's capacity (20480), and lists of equal depths below 2048 (its merge-sort fallback)."""
import numpy as np
import pytest
import torch

from tests.scene_helpers import rects_scene
from tests.test_gpu_sort import _bin_lists, _check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lr():
    import paper_2405_13364_gb300 as P
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    P.load_library()
    return P


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 256, 257, 511, 512, 513, 768, 769, 1024, 1025, 2046, 2047, 2048,
                               2049, 20479, 20480, 20481])
def test_list_length(lr, n):
    # squares inside the image at distinct depths
    rng = np.random.default_rng(n)
    xy = rng.uniform(2, 20, (n, 2))
    rects = [(float(x), float(y), float(x + 3.0), float(y + 2.0)) for x, y in xy]
    s = rects_scene(rects, width=32, height=32, depths=rng.uniform(1.0, 2.0, n),
                    colors=np.concatenate([rng.random((n, 3)), np.full((n, 1), 0.05)], 1))
    st, bin_off, refs, rect = _bin_lists(lr, s)
    lens = _check(s, st, bin_off, refs, rect)
    assert lens.sum() == n
    assert st["bins_high"] == (n >= 2048) and st["sort_bins"] == [int(2048 <= n <= 20480), 0, int(n > 20480)]


@pytest.mark.parametrize("n", [64, 65, 130, 700, 1500, 2047])
def test_equal_depths_below_high_density(lr, n):
    # one depth: a single bucket; from 65 references on the merge sort orders them by index
    rng = np.random.default_rng(n)
    xy = np.floor(rng.uniform(0, 24, (n, 2)) * 4) / 4
    rects = [(float(x), float(y), float(x + 6.0), float(y + 5.0)) for x, y in xy]
    s = rects_scene(rects, width=32, height=32, colors=np.concatenate([rng.random((n, 3)), np.full((n, 1), 0.1)], 1))
    st, bin_off, refs, rect = _bin_lists(lr, s)
    assert _check(s, st, bin_off, refs, rect).sum() == n


def test_many_bins_of_mixed_length(lr):
    # a few bins past 2048 references among many short ones: whole CTAs, then their quarters
    import scenegen
    s = scenegen.gaussian_particles(60_000, 320, 256, seed=9, sigma=0.6, size_px=(2.0, 8.0))
    st, bin_off, refs, rect = _bin_lists(lr, s)
    lens = _check(s, st, bin_off, refs, rect)
    assert st["bins_high"] > 0 and (lens < 2048).sum() > 20
