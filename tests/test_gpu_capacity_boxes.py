"""Slots that exceed a capacity in a launch of more blocks than fit the GPU at
once, so that blocks of a slot start when its last chunk is done: the depth boxes
listed for them (Sec. II-D-1) leave the slots' next frames with the oracle's depth
images, whichever value of the slot's size those blocks saw."""
import math

import numpy as np
import pytest
import torch

from synth import render
from synth.scenes import _gen, _make_rig, player
from tests.gpu_harness import compare, fetch_outputs, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "the -m gpu tests need a CUDA GPU"
    from paper_1903_11785_gb300.build import build
    build()


@pytest.mark.parametrize("n,capacity", [(5, "max_verts"), (40, "max_tris")])
def test_frames_after_an_overflow(n, capacity):
    from paper_1903_11785_gb300 import fvv
    cs = [(8 * math.cos(2 * math.pi * (k + 0.2) / n), 8 * math.sin(2 * math.pi * (k + 0.2) / n), 3.0) for k in range(n)]
    rig = _make_rig("overflow", cs, [(0.0, 0.0, 0.9)] * n, 190.0, 240, 150, _gen(f"overflow/{n}"), (-3.0, -3.0, 0.0),
                    (3.0, 3.0, 2.3), 0.12, 0.05, 3)
    g = _gen("overflow/players")
    one = player((0.0, 0.0), 0.3, 1.8, g, 0)
    crowd = sum((player((-1.2 + 0.8 * k, 0.4 * (-1) ** k), 0.3 * k, 1.8, g, k) for k in range(4)), [])
    small, large = (render(rig, objs, index=i, config_tag="overflow", flip_prob=0.0) for i, objs in enumerate((one, crowd)))
    ref = run_oracle(rig, small)
    need = {"max_verts": len(ref[0].verts), "max_tris": len(ref[0].tris)}[capacity]
    slots = list(range(96))
    r = fvv.Rig(rig, max_slots=len(slots), host_staging=0, max_fine_words=1 << 16, **{capacity: need})
    try:
        for over in (large, small, large, large, small):
            for s in slots:
                fr = over if s % 3 else small
                r.upload_silhouettes(s, fr.masks.cuda())
            r.reconstruct(slots)
            r.colour(slots, [small.rgb.cuda()] * len(slots), np.stack([small.viewpoint] * len(slots)))
            torch.cuda.synchronize()
            for s in (0, 1, 50, 51, 94, 95):
                o = fetch_outputs(r, s)
                if s % 3 and over is large:
                    assert o["counts"]["flags"] & {"max_verts": 1 << 3, "max_tris": 1 << 4}[capacity]   # FVV_FLAG_*
                    assert o["counts"]["n_verts"] == 0
                else:
                    compare(rig, small, o, ref)
    finally:
        r.close()
