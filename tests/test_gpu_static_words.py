"""The allocation-free render's pair count comes through pinned words that its calls
share, whatever the camera: calls from several threads, one at a time, each get their
own count, and creating a camera allocates its ray tables alone."""
import dataclasses
import threading

import pytest

from paper_2510_12901_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def test_threads_taking_turns():
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    views = []
    for i, (n, w, h) in enumerate([(4096, 64, 64), (1, 17, 9), (20000, 64, 48), (6000, 33, 65)]):
        cam = dataclasses.replace(syn.tiny_camera(), width=w, height=h, cx=w / 2, cy=h / 2)
        views.append((sg.Scene(syn.tiny_scene(seed=90 + i, n=n)), sg.Camera(cam), cam))

    def render(k, st):
        S, C, cam = views[k]
        o = [torch.full(s, float("nan"), device="cuda")
             for s in ((cam.height, cam.width, 3), (cam.height, cam.width), (cam.height, cam.width))]
        sg.sg_render_camera_static(S.handle, C.handle, cam.c2w, sg.sg_default_opts(),
                                   *[t.data_ptr() for t in o], st.cuda_stream)
        st.synchronize()
        return o

    want = [render(k, torch.cuda.current_stream()) for k in range(len(views))]
    assert float(want[0][1].max()) > 0.5
    lock, bad = threading.Lock(), []

    def work(t):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for i in range(16):
                k = (i * (t + 1) + t) % len(views)
                with lock:
                    got = render(k, st)
                if not all(torch.equal(a, b) for a, b in zip(got, want[k])):
                    bad.append((t, i, k))

    ts = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad[:5]


def test_a_camera_allocates_its_tables_alone():
    from paper_2510_12901_gb300 import simgut as sg
    cam = syn.tiny_camera()
    sg.Camera(cam)
    n = sg.sg_alloc_count()
    c = sg.Camera(cam)
    # four tables (rays, tangent-plane rays, tile directions and bases) and three
    # arrays freed again
    assert sg.sg_alloc_count() - n == 4 + 2 * 3
    del c
    assert sg.sg_alloc_count() - n == 2 * 7
