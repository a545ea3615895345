"""The pair count reaches the host through pinned words that the offsets kernel
writes, behind a sequence number of the frame's renders.  Frames that change
scene, size and mode between renders, and frames rendered by several threads on
streams of their own, must each see their own count."""
import dataclasses
import threading

import numpy as np
import pytest

from paper_2510_12901_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def _scenes(sg):
    cam = syn.tiny_camera()
    away = syn.tiny_scene(seed=3, n=100)
    away.means[:, 1] -= 50.0                      # behind the camera: no pair
    return [(sg.Scene(sc), sg.Camera(dataclasses.replace(cam, width=w, height=h)), cam.c2w)
            for sc, w, h in ((syn.tiny_scene(seed=1, n=4096), 64, 64), (away, 64, 64),
                             (syn.tiny_scene(seed=2, n=1), 17, 9),
                             (syn.tiny_scene(seed=4, n=20000), 64, 48))]


def _render(sg, view, frame, stream=None):
    import torch
    S, C, c2w = view
    o = sg.render_camera(S, C, c2w, frame=frame, stream=stream)
    if stream is None:
        torch.cuda.synchronize()
    else:
        stream.synchronize()
    return frame.stats()[0], o["rgb"].cpu().numpy()


def test_one_frame_many_views():
    from paper_2510_12901_gb300 import simgut as sg
    views = _scenes(sg)
    want = [_render(sg, v, sg.Frame()) for v in views]
    assert want[1][0] == 0 and want[0][0] > 0
    fr = sg.Frame()
    for k, i in enumerate([0, 1, 3, 2, 0, 0, 3, 1, 1, 2]):
        if k == 5:      # a render that leaves the count on the device
            sg.sg_frame_set_capacity(fr.handle, 1 << 20)
            assert _render(sg, views[i], fr)[0] == want[i][0]
            sg.sg_frame_set_capacity(fr.handle, 0)
        n, rgb = _render(sg, views[i], fr)
        assert n == want[i][0]
        assert np.array_equal(rgb, want[i][1])


def test_threads_with_frames_and_streams():
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    views = _scenes(sg)
    want = [_render(sg, v, sg.Frame()) for v in views]
    bad = []

    def work(t):
        st, fr = torch.cuda.Stream(), sg.Frame()
        for k in range(24):
            i = (k * (t + 1) + t) % len(views)
            with torch.cuda.stream(st):
                n, rgb = _render(sg, views[i], fr, st)
            if n != want[i][0] or not np.array_equal(rgb, want[i][1]):
                bad.append((t, k, i, n))

    ts = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad[:5]
