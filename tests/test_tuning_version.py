"""Launch shapes that the autotuner's cache (paper_1903_11785_gb300/tuning_cache.py)
stored for earlier kernels, when "zbuffer_cams" counted cameras a block, are not
applied: the workload is tuned again and stored beside them."""
import json

from paper_1903_11785_gb300 import tuning_cache as tc
from synth import make_rig
from tests.test_tuning_cache import SHAPES, FakeRig


def test_shapes_of_earlier_kernels_are_left_alone(tmp_path):
    path, v = str(tmp_path / "tuning.json"), make_rig("volleyball")
    key = tc.workload_key(v, 2, "NVIDIA GB300")
    old = "v1|" + key.split("|", 1)[1]
    stored = dict(SHAPES, zbuffer_cams=1, fine=(64, 2))
    tc.store(path, old, stored)
    rig = FakeRig()
    shapes, cached = tc.tuned(rig, v, [0, 1], path, "NVIDIA GB300")
    assert not cached and shapes == SHAPES and rig.calls == [("autotune", (0, 1))]
    assert set(json.load(open(path))) == {old, key} and tc.lookup(path, old) == stored
