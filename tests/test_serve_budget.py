"""The serving loop's memory budget (Sec. III-B: the memory is taken at start-up):
the arenas of all the library rigs that a Server makes stay within it.  Stand-ins
take the place of fvv.Rig, the fitting pass and the streams, so no GPU is needed;
the arenas' sizes are fvv_query_arena's."""
import numpy as np
import pytest
import torch

from synth import make_rig


@pytest.fixture
def serve(monkeypatch):
    from paper_1903_11785_gb300.build import build
    build()
    from paper_1903_11785_gb300 import fvv, serve as mod

    class FakeRig:
        made = []

        def __init__(self, scene_rig, max_slots, host_staging, **caps):
            self.arena_bytes = fvv.fvv_query_arena(fvv.make_desc(scene_rig, max_slots, host_staging),
                                                   fvv.make_params(scene_rig, **caps))
            FakeRig.made.append(self)

    monkeypatch.setattr(mod.fvv, "Rig", FakeRig)
    monkeypatch.setattr(mod, "fitted_caps", lambda pool, staging, base: dict(base, max_fine_words=1 << 17))
    monkeypatch.setattr(torch.cuda, "Stream", lambda *a, **k: None)
    mod.made = FakeRig.made
    return mod


def _pool(serve, config):
    rig = make_rig(config)
    some = [torch.zeros(1, dtype=torch.uint8)]
    return serve.RigPool(scene_rig=rig, masks=some, rgb=some, viewpoints=np.zeros((1, 3), np.float32))


@pytest.mark.parametrize("fit", [True, False])
@pytest.mark.parametrize("configs", [("volleyball",), ("volleyball", "judo", "volleyball")])
def test_all_arenas_stay_within_the_budget(serve, configs, fit):
    pools = [_pool(serve, c) for c in configs]
    caps = dict(max_fine_words=1 << 18)
    for budget in (6 << 30, 9 << 30, 20 << 30):
        del serve.made[:]
        srv = serve.Server(pools, budget_bytes=budget, max_slots_per_group=1000, caps=caps, fit_caps=fit)
        groups = len(set(configs))
        assert len(serve.made) == groups * (2 if fit else 1) and min(srv.slots) >= 1
        used = sum(r.arena_bytes for r in serve.made)
        # within the budget, and no more than a slot of each group below it
        assert budget - groups * max(g.slot_bytes for g in srv.groups) <= used <= budget
