"""The backward that writes its gradients instead of adding them: arrays full of
other values, every feature width, row counts around a block of 128, starts on
and off a 16-byte boundary, blocks without any gradient.  It must give what
adding to zeros gives, 0 in every row without a gradient, and nothing outside
the arrays."""
import numpy as np
import pytest

from paper_2510_12901_gb300 import synthetic as syn
from tests.test_gpu_grad_rows import _scene

pytestmark = pytest.mark.gpu


def _both(sg, shapes, add, write, shift):
    import torch
    got = []
    for call, fill in ((add, 0.0), (write, float("nan"))):
        bufs = [torch.full((int(np.prod(s)) + 8,), 5.0, device="cuda") for s in shapes]
        views = [b[shift:shift + int(np.prod(s))] for b, s in zip(bufs, shapes)]
        for v in views:
            v.fill_(fill)
        call(sg.sg_grads(*[v.data_ptr() for v in views]))
        torch.cuda.synchronize()
        for b, v in zip(bufs, views):
            assert (b[:shift] == 5.0).all() and (b[shift + v.numel():] == 5.0).all()
        got.append([v.cpu().numpy().reshape(s) for v, s in zip(views, shapes)])
    for a, w in zip(*got):
        # the same sums in another order of the atomics: a few roundings of terms
        # that partly cancel
        assert np.abs(a - w).max() <= 1e-4 * max(np.abs(a).max(), 1e-30)
        none = (a == 0).reshape(len(a), -1).all(axis=1)
        assert (w[none] == 0).all()
    return got[0]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("degree", [None, 0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 1003])
def test_camera(n, degree, shift):
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    sc, cam = _scene(n, degree), syn.tiny_camera()
    sc.means[:n // 2, 1] -= 50.0                      # behind the camera: whole blocks without
    S, C, fr = sg.Scene(sc), sg.Camera(cam), sg.Frame()
    o = sg.render_camera(S, C, cam.c2w, frame=fr)
    ups = [torch.ones_like(o[k]) for k in ("rgb", "alpha", "depth")]
    st = torch.cuda.current_stream().cuda_stream
    args = (S.handle, fr.handle, *[u.data_ptr() for u in ups])
    g = _both(sg, [(n, 3), (n, 3), (n, 4), (n,), (n, sc.features.shape[1])],
              lambda gs: sg.sg_backward_camera(*args, gs, st),
              lambda gs: sg.sg_backward_camera_write(*args, gs, st), shift)
    assert np.abs(g[0][-1]).max() > 0


def test_lidar_and_missing_arrays():
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    n = 1500
    L = syn.street_lidar(n_beams=64, n_cols=128)
    sc = syn.street_scene(n, seed=61, kind="lidar", length=60.0)
    S, Ld, fr = sg.Scene(sc), sg.Lidar(L), sg.Frame()
    o = sg.render_lidar(S, Ld, L.col_c2w, frame=fr)
    poses = torch.from_numpy(np.ascontiguousarray(L.col_c2w, np.float32)).cuda()
    o = sg.render_lidar(S, Ld, poses, frame=fr)
    ups = [torch.ones_like(o[k]) for k in ("range", "intensity", "drop", "alpha")]
    st = torch.cuda.current_stream().cuda_stream
    args = (S.handle, fr.handle, *[u.data_ptr() for u in ups])
    _both(sg, [(n, 3), (n, 3), (n, 4), (n,), (n, 3)],
          lambda gs: sg.sg_backward_lidar(*args, gs, st),
          lambda gs: sg.sg_backward_lidar_write(*args, gs, st), 0)
    only = torch.full((n, 3), float("nan"), device="cuda")     # NULL arrays: not wanted
    sg.sg_backward_lidar_write(*args, sg.sg_grads(0, only.data_ptr(), 0, 0, 0), st)
    torch.cuda.synchronize()
    assert torch.isfinite(only).all() and only.abs().max() > 0


def test_autograd_with_one_output_used():
    import torch
    from paper_2510_12901_gb300 import autograd as sga, simgut as sg
    sc, cam = _scene(300, 1), syn.tiny_camera()
    S, C, fr = sg.Scene(sc), sg.Camera(cam), sg.Frame()
    grads = {}
    for k in range(3):
        p = {x: torch.from_numpy(np.array(getattr(sc, x))).cuda().requires_grad_()
             for x in ("means", "log_scales", "quats", "opacity", "features")}
        outs = sga.render_camera(p, S, C, cam.c2w, frame=fr)
        outs[k].sum().backward()
        grads[k] = p["means"].grad
        assert torch.isfinite(grads[k]).all() and grads[k].abs().max() > 0
