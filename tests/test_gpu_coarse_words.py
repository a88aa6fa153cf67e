"""The coarse hull's two passes (Sec. II-B-1) at the edges of their rules, every
output compared with the oracle bit for bit: rows of fewer voxels than a word, of
whole words and of a word and one voxel; fewer cameras than the first pass takes and
more than the table holds; cameras that see part of the volume under both policies;
one frame (three cameras in the first pass) and a batch large enough for one; and
images whose sides no block of the blocked silhouettes divides."""
import math

import numpy as np
import pytest
import torch

from synth import ABSTAIN, STRICT, render, sphere_scene
from synth.scenes import _gen, _make_rig
from tests.gpu_harness import compare, fetch_outputs, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "the -m gpu tests need a CUDA GPU"
    from paper_1903_11785_gb300.build import build
    build()


def _rig(n, nx, ny, nz, focal, policy, W=131, H=93):
    cs = [(9 * math.cos(2 * math.pi * (k + 0.3) / n), 9 * math.sin(2 * math.pi * (k + 0.3) / n), 3.0) for k in range(n)]
    s = 0.1
    rig = _make_rig("words", cs, [(0.0, 0.0, 1.0)] * n, focal, W, H, _gen(f"words/{n}"),
                    (-s * nx / 2, -s * ny / 2, 0.0), (s * nx / 2, s * ny / 2, s * nz), s, s, 2)
    rig.oob_policy = policy
    rig.t_np = 1
    return rig


@pytest.mark.parametrize("nx", [7, 32, 33, 64, 95])
@pytest.mark.parametrize("n,focal,policy", [(1, 100.0, STRICT), (3, 100.0, ABSTAIN), (9, 100.0, STRICT),
                                            (12, 250.0, ABSTAIN)])
def test_rows_and_cameras(nx, n, focal, policy):
    rig = _rig(n, nx, 21, 19, focal, policy)
    fr = render(rig, sphere_scene((0.05, -0.1, 1.0), 0.5), index=n, config_tag="words")
    ref = compare(rig, fr, run_gpu(rig, [fr], caps=dict(max_fine_words=1 << 18))[0])
    assert ref.coarse.sum() > 10


@pytest.mark.parametrize("policy", [STRICT, ABSTAIN])
def test_batch_with_one_camera_in_the_first_pass(policy):
    from paper_1903_11785_gb300 import fvv
    F, rig = 40, _rig(5, 33, 160, 50, 100.0, policy)        # 16,000 words a frame
    frames = [render(rig, sphere_scene((0.05, 0.2 * k, 1.0), 0.5), index=k, config_tag="words") for k in range(2)]
    r = fvv.Rig(rig, max_slots=F, host_staging=0, max_fine_words=1 << 17)
    try:
        for s in range(F):
            r.upload_silhouettes(s, frames[s % 2].masks.cuda())
        r.reconstruct(list(range(F)))
        r.colour(list(range(F)), [frames[s % 2].rgb.cuda() for s in range(F)],
                 np.stack([frames[s % 2].viewpoint for s in range(F)]))
        torch.cuda.synchronize()
        for s in (0, F - 1):
            compare(rig, frames[s % 2], fetch_outputs(r, s))
    finally:
        r.close()
