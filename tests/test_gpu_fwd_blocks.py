"""Blocks an SM of the forward camera compositing: by the size of the render for a
view alone, a fixed number for views of one call on streams of their own.  The image
is the same bit for bit."""
import dataclasses

import pytest

from paper_2510_12901_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


# pairs / tiles on either side of the rule's lines: 4, 6 and 8 blocks for a view alone
@pytest.mark.parametrize("n,w,h", [(3000, 37, 21), (200000, 640, 480), (200000, 1100, 1000)])
def test_same_image_alone_and_beside_another_view(n, w, h):
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    src = syn.street_scene(n, seed=81, sh_degree=1)
    fish, pin = syn.street_cameras(seed=81)
    cam = dataclasses.replace(pin, width=w, height=h, fx=pin.fx * w / pin.width,
                              fy=pin.fy * w / pin.width, cx=w / 2, cy=h / 2)
    S, C, frames = sg.Scene(src), sg.Camera(cam), [sg.Frame() for _ in range(3)]
    for f in frames:
        sg.sg_frame_set_backward_state(f.handle, 0)
    opts = sg.sg_default_opts()
    want = sg.render_camera(S, C, cam.c2w, opts, frame=frames[0])
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    for pick in ((0, 1), (0, 0)):       # streams of their own, one stream
        outs = [[torch.full(s, float("nan"), device="cuda") for s in ((h, w, 3), (h, w), (h, w))]
                for _ in range(2)]
        torch.cuda.synchronize()
        views = sg.sg_camera_views([
            (C.handle, cam.c2w, f.handle, *[t.data_ptr() for t in o], streams[k].cuda_stream)
            for f, k, o in zip(frames[1:], pick, outs)])
        sg.sg_render_cameras(S.handle, views, opts)
        torch.cuda.synchronize()
        for o in outs:
            assert all(torch.equal(a, want[k]) for a, k in zip(o, ("rgb", "alpha", "depth")))
