"""The workspace's size grows with the scene, also where the binning changes its chunks: a workspace that fits
more quads fits fewer."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bin_size", [16, 32, 64])
def test_size_grows_with_quads(bin_size):
    import paper_2405_13364_gb300 as P
    from paper_2405_13364_gb300 import _binding as B
    r = P.Renderer(bin_size=bin_size)
    for w, h in ((64, 64), (1920, 1080)):
        for at in [304 * 2 ** k for k in range(8, 12)] + [400 * 4096, 256, 1024]:   # chunks of 256 ... 4096 quads
            sizes = [B.lr_workspace_size(r.ctx, q, w, h) for q in (at - 257, at - 1, at, at + 1, at + 257) if q >= 0]
            assert sizes == sorted(sizes), (at, sizes)
    r.close()
