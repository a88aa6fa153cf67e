"""fvv_render_view on a stream of its own: its outputs are allocated on the
current stream, so dropping them must not hand their memory out while the
stream still writes it (a second view on another stream would share it)."""
import pytest
import torch

from synth import make_frame

pytestmark = pytest.mark.gpu


def test_dropped_views_on_other_streams_do_not_share_memory():
    from paper_1903_11785_gb300 import fvv
    rig, fr = make_frame("tiny", 0)
    r = fvv.Rig(rig, max_slots=1, host_staging=0)
    try:
        rgb = fr.rgb.cuda()
        r.upload_silhouettes(0, fr.masks.cuda())
        r.reconstruct([0])
        torch.cuda.synchronize()
        a, b = torch.cuda.Stream(), torch.cuda.Stream()
        view = lambda cam, s: r.render_view(0, rgb, rig.P[cam], rig.centre[cam], 3000, 1700, stream=s)  # noqa: E731
        ref = [t.clone() for t in view(1, None)]
        torch.cuda.synchronize()
        for _ in range(20):
            with torch.cuda.stream(a):
                torch.cuda._sleep(2_000_000)         # a's view is still to come when b's is asked for
            ptr = view(0, a)[0].data_ptr()           # dropped at once
            got = view(1, b)
            assert got[0].data_ptr() != ptr
            torch.cuda.synchronize()
            for t, x in zip(got, ref):
                assert torch.equal(t, x)
    finally:
        r.close()
