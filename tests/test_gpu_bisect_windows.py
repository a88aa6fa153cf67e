"""The bisection's sorted windows (Sec. II-C) with the 64-bit camera lists: what a
window keeps of a vertex beside its list (whether its edge is inside every image,
whether some camera saw all of it) for edges inside the images and leaving them,
windows of two and four rows and a last one partly filled; every output compared
with the oracle bit for bit."""
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


@pytest.mark.parametrize("n,focal,fine,policy,rows", [
    (33, 220.0, 0.02, STRICT, 2),       # the sphere inside every image
    (34, 1300.0, 0.05, ABSTAIN, 2),     # and over the images' borders
    (64, 1300.0, 0.03, ABSTAIN, 4),
])
def test_many_cameras_in_sorted_windows(n, focal, fine, policy, rows):
    from paper_1903_11785_gb300 import fvv
    cs = [(5 * math.cos(2 * math.pi * (k + 0.3) / n), 5 * math.sin(2 * math.pi * (k + 0.3) / n), 1.5 + 0.03 * k)
          for k in range(n)]
    rig = _make_rig("windows", cs, [(0.0, 0.0, 1.0)] * n, focal, 310, 246, _gen(f"windows/{n}"), (-1.2, -1.2, 0.0),
                    (1.2, 1.2, 2.2), 0.12, fine, 5)
    rig.oob_policy = policy
    fr = render(rig, sphere_scene((0.1, -0.1, 1.0), 0.6), index=n, config_tag="windows")
    tuning = {k: (256, 8) for k in fvv.TUNE_KNOBS} | {"bisect": (32, 1)}
    g = run_gpu(rig, [fr], tuning=tuning, caps=dict(max_fine_words=1 << 20))[0]
    # one warp a block and one block an SM: windows of k rows from 64 k vertices a warp on
    nv, warps = g["counts"]["n_verts"], torch.cuda.get_device_properties(0).multi_processor_count
    assert next(k for k in (4, 2, 1) if k == 1 or nv >= 64 * warps * k) == rows and nv % (32 * rows) != 0
    compare(rig, fr, g)
