"""The compaction's chunks of one to four turns of 256 fine words (chosen by the
words of all the slots of a launch): a frame with several objects alone and in
launches of more and more slots, where chunks end within and across turns, warps
and objects; every output of the first and last slot against the oracle."""
import math

import numpy as np
import pytest
import torch

from synth import render
from synth.scenes import _gen, _make_rig, player
from tests.gpu_harness import compare, fetch_outputs, run_oracle

pytestmark = pytest.mark.gpu


def test_frames_in_launches_of_many_slots():
    assert torch.cuda.is_available(), "the -m gpu tests need a CUDA GPU"
    from paper_1903_11785_gb300 import fvv
    n = 6
    cs = [(8 * math.cos(2 * math.pi * (k + 0.2) / n), 8 * math.sin(2 * math.pi * (k + 0.2) / n), 3.0) for k in range(n)]
    rig = _make_rig("turns", cs, [(0.0, 0.0, 0.9)] * n, 190.0, 240, 150, _gen("turns"), (-3.0, -3.0, 0.0),
                    (3.0, 3.0, 2.3), 0.12, 0.01, 3)
    g = _gen("turns/players")
    objs = player((-2.0, 1.5), 0.3, 1.8, g, 0) + player((2.1, -1.0), 1.0, 1.7, g, 1) + player((0.2, 2.2), 2.0, 1.9, g, 2)
    fr = render(rig, objs, index=0, config_tag="turns", flip_prob=0.0)
    want = run_oracle(rig, fr)
    slots = 64
    masks, rgb = fr.masks.cuda(), fr.rgb.cuda()
    r = fvv.Rig(rig, max_slots=slots, host_staging=0)
    try:
        for s in range(slots):
            r.upload_silhouettes(s, masks)
        words = 0
        for k in (1, 12, 24, 40, 64):
            r.reconstruct(list(range(k)))
            r.colour(list(range(k)), [rgb] * k, np.stack([fr.viewpoint] * k))
            torch.cuda.synchronize()
            for s in {0, k - 1}:
                out = fetch_outputs(r, s)
                compare(rig, fr, out, want)
                words = out["counts"]["n_fine_words"]
        # the sizes do reach from one turn to the most (152 SMs x 4 blocks x 4 chunks x 256 words a turn)
        assert words < 2 * 622592 and 64 * words > 4 * 622592
    finally:
        r.close()
