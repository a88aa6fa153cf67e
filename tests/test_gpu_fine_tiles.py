"""The fine hull's tiles (Sec. II-B-3) at the edges of their rules, every output
compared with the oracle bit for bit: camera counts on both sides of the lane
groups (8 and 16 lanes a tile, more cameras than lanes), each tile shape on ROIs
whose sides no tile divides, cameras that see only part of the volume (tiles in
part outside an image) under both policies, and silhouettes wide enough that
whole tiles are occupied."""
import math

import pytest
import torch

from synth import ABSTAIN, STRICT, render, sphere_scene
from synth.scenes import _gen, _make_rig
from tests.gpu_harness import compare, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "the -m gpu tests need a CUDA GPU"
    from paper_1903_11785_gb300.build import build
    build()


@pytest.mark.parametrize("tile", [(4, 4, 8), (4, 4, 4), (4, 8, 8)], ids=str)
@pytest.mark.parametrize("n,focal,policy", [(1, 300.0, STRICT), (8, 300.0, STRICT), (9, 300.0, ABSTAIN),
                                            (16, 900.0, ABSTAIN), (17, 300.0, STRICT), (40, 900.0, ABSTAIN)])
def test_tiles_and_lane_groups(n, focal, policy, tile):
    from paper_1903_11785_gb300 import fvv
    cs = [(5 * math.cos(2 * math.pi * (k + 0.3) / n), 5 * math.sin(2 * math.pi * (k + 0.3) / n), 2.0 + 0.1 * k)
          for k in range(n)]
    # a focal length of 900 leaves part of the sphere outside each image
    rig = _make_rig("tiles", cs, [(0.0, 0.0, 1.0)] * n, focal, 330, 250, _gen(f"tiles/{n}"), (-1.5, -1.5, 0.0),
                    (1.5, 1.5, 2.2), 0.11, 0.031, 4)
    rig.oob_policy = policy
    fr = render(rig, sphere_scene((0.1, -0.2, 1.0), 0.6), index=n, config_tag="tiles")
    tuning = {k: (256, 8) for k in fvv.TUNE_KNOBS} | {"fine_tile": tile}
    ref = compare(rig, fr, run_gpu(rig, [fr], tuning=tuning, caps=dict(max_fine_words=1 << 19))[0])
    assert len(ref.tris) > 1000
