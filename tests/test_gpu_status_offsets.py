"""A wait of the pair-offsets scan that gives up is told with the pair count, also
where the last tile need not wait itself: with more than 32 tiles it can take its
prefix from a tile whose own wait gave up."""
import numpy as np
import pytest

from paper_2510_12901_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


# tiles of 2048 entries up to 262144 Gaussians, of 8192 above
@pytest.mark.parametrize("n,hold", [(150000, 0), (150000, 31), (150000, 70), (300000, 0)])
def test_offsets_timeout_with_many_tiles(n, hold):
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    sc = syn.tiny_scene(seed=51, n=n)
    sc.means[:, 1] = np.random.default_rng(52).uniform(-8.0, 10.0, n)
    sc.means[:, [0, 2]] *= 0.05 * (sc.means[:, 1:2] + 10.0)     # in view
    sc.log_scales -= 1.0
    cam = syn.tiny_camera()
    S, C, fr = sg.Scene(sc), sg.Camera(cam), sg.Frame()
    ref = sg.render_camera(S, C, cam.c2w, frame=fr)
    torch.cuda.synchronize()
    visible = int((fr.field(sg.FIELD_COUNT, np.uint32) > 0).sum())
    assert visible > (8192 if n > 262144 else 2048) * max(hold + 2, 33)
    try:
        for _ in range(10):
            sg.sg_debug_lookback(200, sg.LOOKBACK_OFFSETS, hold)
            with pytest.raises(sg.SimgutError) as e:
                sg.render_camera(S, C, cam.c2w, frame=fr)
            assert e.value.status == -5 and "gave up" in str(e.value)
    finally:
        sg.sg_debug_lookback(0, sg.LOOKBACK_NONE, -1)
    out = sg.render_camera(S, C, cam.c2w, frame=fr)
    sg.sg_frame_status(fr.handle)
    assert all(torch.equal(out[k], ref[k]) for k in ("rgb", "alpha", "depth"))
