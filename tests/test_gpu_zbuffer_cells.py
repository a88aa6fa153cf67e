"""The z-buffer's pixel cells (Sec. II-D-1): the bytewise test that turns
(triangle, camera) pairs away before they are drawn must keep every pair that
covers a pixel.  Rigs at the edges of that rule, every output compared with the
oracle bit for bit: meshes of sub-pixel and of many-pixel triangles, a camera
whose cells may be 64 pixels or more (its cells do not decide), a camera inside
the volume (no bound on w'), camera counts that leave a group of four
incomplete, and both ways of sharing a frame's triangles among the warps."""
import math

import pytest
import torch

from synth import ABSTAIN, render, scene_objects
from synth.scenes import _gen, _make_rig, look_at_camera
from tests.gpu_harness import compare, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "the -m gpu tests need a CUDA GPU"
    from paper_1903_11785_gb300.build import build
    build()


def _rig(n, fine, focal, first=None, centre=None):
    """n cameras around the tiny scene; camera 0 with focal length `first` or at `centre`."""
    g = _gen(f"cells/{n}/{fine}/{focal}/{first}")
    cs = [(6 * math.cos(2 * math.pi * (k + 0.2) / n), 6 * math.sin(2 * math.pi * (k + 0.2) / n), 3.0) for k in range(n)]
    if centre is not None:
        cs[0] = centre
    rig = _make_rig("cells", cs, [(0.0, 0.0, 0.9)] * n, focal, 640, 360, g, (-2.0, -2.0, 0.0), (2.0, 2.0, 2.5),
                    max(0.05, 2 * fine), fine, 6)
    if first is not None:
        obj = scene_objects("tiny", 0)
        K, R, P = look_at_camera(cs[0], obj[2].centre, first, 640, 360)
        rig.K64[0], rig.R64[0], rig.P64[0] = K, R, P
        rig.P[0] = P.astype("float32")
    rig.oob_policy = ABSTAIN
    return rig


@pytest.mark.parametrize("n,fine,focal,first,centre,quads", [
    (5, 0.01, 60.0, None, None, 4),       # a pixel holds many triangles
    (7, 0.04, 500.0, None, None, 1),      # triangles of a few pixels
    (5, 0.05, 500.0, 4000.0, None, 4),    # camera 0: triangles of about 30 pixels, cells still decide
    (5, 0.05, 500.0, 9000.0, None, 2),    # camera 0: a cell may span 64 pixels, its cells do not decide
    (6, 0.02, 400.0, None, (0.3, 0.2, 1.4), 4),   # camera 0 inside the volume
    (1, 0.02, 500.0, None, None, 4),
    (17, 0.03, 300.0, None, None, 4),     # five groups of four, the last with one camera
])
def test_pairs_kept_by_pixel_cells(n, fine, focal, first, centre, quads):
    from paper_1903_11785_gb300 import fvv
    rig = _rig(n, fine, focal, first, centre)
    fr = render(rig, scene_objects("tiny", 0), index=0, config_tag="cells")
    tuning = {k: (128, 4) for k in fvv.TUNE_KNOBS} | {"zbuffer_cams": quads, "zbuffer": (64, 1)}
    caps = dict(max_fine_words=1 << 20)
    for t in (None, tuning):              # many warps for few triangles, and few warps
        assert len(compare(rig, fr, run_gpu(rig, [fr], tuning=t, caps=caps)[0]).tris) > 100
