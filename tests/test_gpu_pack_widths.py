"""Packing of masks whose rows start at any address: widths that 4, 16 and 32 do
and do not divide, images of one row and of few pixels, masks that begin 0 to 3
bytes into a buffer, in device memory and in place in pinned host memory.  Every
bit against the mask itself; the bytes around a mask are set, so that none of them
is taken for it."""
import dataclasses

import numpy as np
import pytest
import torch

from synth import make_rig
from tests.gpu_harness import unpack_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("W,H", [(1, 1), (3, 2), (31, 7), (32, 5), (33, 4), (36, 9), (61, 3), (64, 1), (630, 6), (1277, 11)])
def test_every_bit_at_every_start(W, H, host):
    assert torch.cuda.is_available(), "the -m gpu tests need a CUDA GPU"
    from paper_1903_11785_gb300 import fvv
    tiny = make_rig("tiny")
    n = tiny.n_cams
    rig = dataclasses.replace(tiny, width=np.full(n, W, np.int32), height=np.full(n, H, np.int32))
    g = np.random.default_rng(W * 100 + H)
    r = fvv.Rig(rig, max_slots=1, host_staging=0, max_fine_words=1 << 16, max_verts=1024, max_tris=1024)
    try:
        for start in range(4):
            masks = ((g.random((n, H, W)) < 0.4) * g.integers(1, 256, (n, H, W))).astype(np.uint8)
            buf = torch.full((start + masks.size + 64,), 255, dtype=torch.uint8)
            buf[start:start + masks.size] = torch.from_numpy(masks.reshape(-1))
            buf = buf.pin_memory() if host else buf.cuda()
            r.upload_silhouettes(0, buf[start:start + masks.size].view(n, H, W), in_place=host)
            torch.cuda.synchronize()
            sil = r.debug(0, fvv.FVV_DEBUG_SIL_BITS).cpu().numpy().view(np.uint32)
            np.testing.assert_array_equal(unpack_rows(sil, (n, H), W), (masks != 0).astype(np.uint8))
    finally:
        r.close()
