"""Depth images cleared by object (Sec. II-D-1) for frames of up to 150 objects, more
than the 32 boxes a warp of the clear takes at a time: apart, where each is cleared by
itself, or crowded in an image's corner, where their common box is; a slot that holds
many, few, none and many again has the oracle's whole depth images each time."""
import math

import numpy as np
import pytest
import torch

from synth import render, sphere_scene
from synth.scenes import _gen, _make_rig
from tests.gpu_harness import compare, fetch_outputs, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "the -m gpu tests need a CUDA GPU"
    from paper_1903_11785_gb300.build import build
    build()


def _balls(nx, ny, nz, step, r):
    return sum((sphere_scene((step * (i - nx / 2 + 0.5), step * (j - ny / 2 + 0.5), 0.4 + step * k), r)
                for i in range(nx) for j in range(ny) for k in range(nz)), [])


# from above, so that balls side by side stay apart in the images, and from the side, where they do not
@pytest.mark.parametrize("n,height", [(3, 9.0), (3, 1.2), (13, 9.0)])
def test_many_objects(n, height):
    from paper_1903_11785_gb300 import fvv
    cs = [(6 * math.cos(2 * math.pi * (k + 0.2) / n), 6 * math.sin(2 * math.pi * (k + 0.2) / n), height) for k in range(n)]
    rig = _make_rig("many", cs, [(0.0, 0.0, 0.9)] * n, 200.0, 250, 170, _gen(f"many/{n}"), (-2.4, -2.4, 0.0),
                    (2.4, 2.4, 1.6), 0.08, 0.04, 3)
    rig.t_np = 1
    scenes = [_balls(10, 10, 1, 0.44, 0.1), _balls(2, 1, 1, 0.5, 0.1), [], _balls(6, 6, 1, 0.3, 0.08),
              _balls(12, 12, 1, 0.38, 0.07), _balls(6, 5, 1, 0.44, 0.1)]
    frames = [render(rig, s, index=i, config_tag="many", flip_prob=0.0) for i, s in enumerate(scenes)]
    refs = [run_oracle(rig, fr) for fr in frames]
    assert max(len(ref[0].rois) for ref in refs) > 32
    for slots in (1, 9):
        r = fvv.Rig(rig, max_slots=slots, host_staging=0, max_fine_words=1 << 18, max_rois=512)
        try:
            for order in ((0, 1, 4, 2, 3, 5), (3, 0, 2, 4, 1, 0)):
                for j in range(len(order)):
                    now = [frames[order[(j + s) % len(order)]] for s in range(slots)]
                    for s, fr in enumerate(now):
                        r.upload_silhouettes(s, fr.masks.cuda())
                    r.reconstruct(list(range(slots)))
                    r.colour(list(range(slots)), [fr.rgb.cuda() for fr in now], np.stack([fr.viewpoint for fr in now]))
                    torch.cuda.synchronize()
                    for s in {0, slots - 1}:
                        i = order[(j + s) % len(order)]
                        compare(rig, frames[i], fetch_outputs(r, s), refs[i])
        finally:
            r.close()
