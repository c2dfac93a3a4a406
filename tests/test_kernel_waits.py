"""Programmatic dependent launch: every kernel launched that way waits for its predecessor before
anything else, since only the wait makes an earlier grid's writes visible to it; and renders that
reuse one workspace for ever other scenes, small flat views beside a large one, see no stale list."""
import glob
import os
import re

import numpy as np
import pytest
import torch

import scenegen

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_13364_gb300", "csrc")


def _sources():
    out = {}
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(f) as h:
            out[os.path.basename(f)] = re.sub(r"//[^\n]*", "", h.read())
    return out


def test_every_dependent_kernel_waits_first():
    src = _sources()
    text = "\n".join(src.values())
    launched = set(re.findall(r"launch_pdl\(\s*\w+,\s*(k_\w+)", text))
    assert {"k_init", "k_setup", "k_bin_count", "k_bin_sort", "k_raster_ordered", "k_raster", "k_overflow",
            "k_resolve"} <= launched
    first = dict(re.findall(r"\b(k_\w+)\([^;{}]*\)\s*\{\s*([^;]*;)", text))
    assert {k: first.get(k) for k in launched} == {k: "pdl_begin();" for k in launched}
    assert re.search(r"void pdl_begin\(\) \{\s*asm volatile\(\"griddepcontrol\.wait;\" ::: \"memory\"\);", text)
    # and nowhere later or under a condition
    assert text.count("griddepcontrol.wait") == text.count("griddepcontrol.launch_dependents") == 1


@pytest.mark.gpu
@pytest.mark.parametrize("k", [1, 3])
def test_reused_workspace(k):
    import paper_2405_13364_gb300 as P
    r = P.Renderer(sorter_k=k)
    plain = P.Renderer(sorter_k=k)
    for i in range(12):
        rng = np.random.default_rng(i)
        sizes = [(int(rng.integers(8, 90)), int(rng.integers(8, 90))) for _ in range(3)]
        scenes = [scenegen.gaussian_particles(int(rng.integers(50, 900)), w, h, seed=3 * i + n)
                  for n, (w, h) in enumerate(sizes)]
        scenes.insert(int(rng.integers(0, 4)), scenegen.wavy_layers(640, 360, layers=8, nx=40, ny=20, seed=i))
        items = [(P.DeviceScene.from_scene(s), s.width, s.height) for s in scenes]
        got = r.render_batch(items, check=False)
        # with the coverage hash every bin takes the per-pixel sorter
        ref = plain.render_batch(items, hash=True)
        torch.cuda.synchronize()
        for g, e in zip(got, ref):
            assert torch.equal(g["rgba"], e["rgba"])
    r.close()
    plain.close()
