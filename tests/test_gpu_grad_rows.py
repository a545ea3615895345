"""The rows of the gradient arrays: Gaussian counts around a block of 128, every
feature width, arrays that start on a 16-byte boundary or 4 bytes past one.
The gradients are added to what the arrays hold, a second backward of the same
render adds them again (the accumulator starts clear each time), and they
match the oracle's."""
import numpy as np
import pytest

from paper_2510_12901_gb300 import synthetic as syn
from tests.test_gpu_backward import NAMES, compare_grads, upstream

pytestmark = pytest.mark.gpu


def _scene(n, degree):
    sc = syn.tiny_scene(seed=51, n=n)
    if degree is not None:
        rng = np.random.default_rng(52)
        sc.features = rng.normal(0.0, 0.3, (n, 3 * (degree + 1) ** 2)).astype(np.float32)
        sc.feature_kind, sc.sh_degree = syn.FEATURES_SH, degree
    sc.means[-1] = [0.0, -5.0, 0.0]          # the last row always has a gradient
    sc.log_scales[-1] = [0.0, -0.5, 0.3]
    sc.opacity[-1] = 0.7
    return sc


@pytest.mark.parametrize("degree", [None, 0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 1003])
def test_rows_of_every_width_and_alignment(n, degree):
    import torch
    from oracle import Oracle
    from paper_2510_12901_gb300 import simgut as sg
    sc, cam = _scene(n, degree), syn.tiny_camera()
    O = Oracle(64)
    g = upstream(O.render_camera(sc, cam), np.random.default_rng(53))
    Go = O.backward_camera(sc, cam, *g)
    S, C, fr = sg.Scene(sc), sg.Camera(cam), sg.Frame()
    sg.render_camera(S, C, cam.c2w, frame=fr)
    ups = [torch.from_numpy(u).cuda() for u in g]
    shapes = [(n, 3), (n, 3), (n, 4), (n,), (n, sc.features.shape[1])]
    for shift in (0, 1):
        bufs = [torch.full((int(np.prod(s)) + 8,), 5.0, device="cuda") for s in shapes]
        views = [b[shift:shift + int(np.prod(s))].view(s) for b, s in zip(bufs, shapes)]
        for v in views:
            v.zero_()
        gs = sg.sg_grads(*[v.data_ptr() for v in views])
        stream = torch.cuda.current_stream().cuda_stream
        sg.sg_backward_camera(S.handle, fr.handle, *[u.data_ptr() for u in ups], gs, stream)
        once = [v.clone() for v in views]
        sg.sg_backward_camera(S.handle, fr.handle, *[u.data_ptr() for u in ups], gs, stream)
        torch.cuda.synchronize()
        compare_grads(dict(zip(NAMES, [v.cpu().numpy() for v in once])), Go,
                      f"n={n} degree={degree} shift={shift}")
        for a, b in zip(once, views):       # twice, up to the order of the atomics
            assert torch.allclose(b, 2.0 * a, rtol=1e-4, atol=1e-5 * float(a.abs().max()))
        for b, s in zip(bufs, shapes):      # nothing outside the rows
            m = int(np.prod(s))
            assert (b[:shift] == 5.0).all() and (b[shift + m:] == 5.0).all()
