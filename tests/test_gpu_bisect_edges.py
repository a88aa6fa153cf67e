"""The bisection's edge checks (Sec. II-C) at the edges of their rules, every
output compared with the oracle bit for bit: edges of a fraction of a pixel, of
several pixels and of more than the 32 x 8 pixels that are scanned; edges that leave
the image (the general form of the midpoint tests) under both policies; more
than 32 cameras (the 64-bit camera lists); and no steps."""
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


@pytest.mark.parametrize("n,focal,fine,steps,policy", [
    (6, 40.0, 0.02, 7, STRICT),         # a tenth of a pixel an edge
    (6, 400.0, 0.05, 7, STRICT),        # about four pixels an edge
    (6, 2600.0, 0.1, 5, ABSTAIN),       # about 50 pixels an edge, most of the sphere outside every image
    (7, 700.0, 0.06, 6, STRICT),        # the sphere reaches over the images' borders
    (7, 700.0, 0.06, 6, ABSTAIN),
    (33, 300.0, 0.06, 30, STRICT),
    (64, 300.0, 0.08, 4, ABSTAIN),
    (5, 300.0, 0.04, 0, STRICT),
])
def test_edges(n, focal, fine, steps, policy):
    from paper_1903_11785_gb300 import fvv
    cs = [(5 * math.cos(2 * math.pi * (k + 0.3) / n), 5 * math.sin(2 * math.pi * (k + 0.3) / n), 1.5 + 0.03 * k)
          for k in range(n)]
    rig = _make_rig("edges", cs, [(0.0, 0.0, 1.0)] * n, focal, 310, 246, _gen(f"edges/{n}"), (-1.2, -1.2, 0.0),
                    (1.2, 1.2, 2.2), 0.12, fine, steps)
    rig.oob_policy = policy
    fr = render(rig, sphere_scene((0.1, -0.1, 1.0), 0.6), index=n, config_tag="edges")
    one = {k: (256, 8) for k in fvv.TUNE_KNOBS}
    for t in (one, one | {"bisect": (32, 1)}):      # a vertex per lane; few warps, so sorted windows where there is enough
        ref = compare(rig, fr, run_gpu(rig, [fr], tuning=t, caps=dict(max_fine_words=1 << 18))[0])
        assert len(ref.tris) > 20
