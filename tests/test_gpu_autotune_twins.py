"""lr_config.block_h = 4 and 8 take the same kernels: the autotuner renders and times each candidate once
for both, and never picks one of the two by noise."""
import pytest

import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block_hs", [(4, 8), (8, 4)])
def test_twins(block_hs, monkeypatch):
    import paper_2405_13364_gb300 as P
    from paper_2405_13364_gb300 import autotune
    made = []

    class Counted(P.Renderer):
        def __init__(self, *a, **kw):
            made.append(kw)
            super().__init__(*a, **kw)

    monkeypatch.setattr(P, "Renderer", Counted)
    s = scenegen.wavy_layers(160, 90, layers=8, nx=24, ny=12, seed=3)
    res = autotune.tune(P.DeviceScene.from_scene(s), s.width, s.height, ks=(1, 3, 8), reps=3, use_cache=False,
                        bin_sizes=(16, 32), block_hs=block_hs)
    assert len(made) == 3 * 2 and len(res["table"]) == 3 * 2 + 2 * 2
    by = {}
    for t in res["table"]:
        by.setdefault((t["sorter_k"], t["bin_size"]), set()).add(t["ms"])
    assert all(len(v) == 1 for v in by.values())
    assert res["block_h"] == 4
