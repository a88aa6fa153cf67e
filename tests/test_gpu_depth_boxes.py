"""The depth images are cleared where the slot's last z-buffer may have written
(Sec. II-D-1), one box per object and camera: a slot reconstructed with other frames,
an empty one and a frame whose objects' boxes overlap among them, holds the
oracle's whole depth images every time; with enough blocks for every camera and
with fewer blocks than cameras."""
import math

import numpy as np
import pytest
import torch

from synth import render
from synth.scenes import _gen, _make_rig, player
from tests.gpu_harness import compare, fetch_outputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "the -m gpu tests need a CUDA GPU"
    from paper_1903_11785_gb300.build import build
    build()


@pytest.mark.parametrize("n,slots", [(5, 1), (40, 40)])
def test_slot_reuse_with_several_objects(n, slots):
    from paper_1903_11785_gb300 import fvv
    cs = [(8 * math.cos(2 * math.pi * (k + 0.2) / n), 8 * math.sin(2 * math.pi * (k + 0.2) / n), 3.0) for k in range(n)]
    rig = _make_rig("boxes", cs, [(0.0, 0.0, 0.9)] * n, 190.0, 240, 150, _gen(f"boxes/{n}"), (-3.0, -3.0, 0.0),
                    (3.0, 3.0, 2.3), 0.12, 0.05, 3)
    g = _gen("boxes/players")
    one = player((0.0, 0.0), 0.3, 1.8, g, 0)
    spread = player((-2.0, 1.5), 0.3, 1.8, g, 0) + player((2.1, -1.0), 1.0, 1.7, g, 1) + player((0.2, 2.2), 2.0, 1.9, g, 2)
    crowd = sum((player((-1.2 + 0.8 * k, 0.4 * (-1) ** k), 0.3 * k, 1.8, g, k) for k in range(4)), [])
    frames = [render(rig, objs, index=i, config_tag="boxes", flip_prob=0.0)
              for i, objs in enumerate((spread, one, [], crowd, spread))]
    r = fvv.Rig(rig, max_slots=slots, host_staging=0, max_fine_words=1 << 16)
    try:
        every = list(range(slots))
        for fr in frames:
            masks, rgb = fr.masks.cuda(), fr.rgb.cuda()
            for s in every:
                r.upload_silhouettes(s, masks)
            r.reconstruct(every)
            r.colour(every, [rgb] * slots, np.stack([fr.viewpoint] * slots))
            torch.cuda.synchronize()
            compare(rig, fr, fetch_outputs(r, slots - 1))
    finally:
        r.close()
