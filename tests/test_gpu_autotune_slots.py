"""fvv_autotune runs stages again on the slots it is given (the coarse hull
many times, then the ROI table for each tile shape): the slots it is not given keep
every output, and its own end as one reconstruction leaves them."""
import numpy as np
import pytest
import torch

from synth import make_frame, make_rig
from tests.gpu_harness import compare, fetch_outputs

pytestmark = pytest.mark.gpu


def test_autotune_leaves_other_slots_alone():
    from paper_1903_11785_gb300.build import build
    build()
    from paper_1903_11785_gb300 import fvv
    rig = make_rig("hd720")
    frames = [make_frame("hd720", i, rig=rig)[1] for i in range(3)]
    r = fvv.Rig(rig, max_slots=3, host_staging=0)
    try:
        for s, fr in enumerate(frames):
            r.upload_silhouettes(s, fr.masks.cuda())
        r.reconstruct([0, 1, 2])
        r.autotune([1])
        rgb = [fr.rgb.cuda() for fr in frames]
        r.colour([0, 1, 2], rgb, np.stack([fr.viewpoint for fr in frames]))
        torch.cuda.synchronize()
        for s, fr in enumerate(frames):
            compare(rig, fr, fetch_outputs(r, s))
    finally:
        r.close()
