"""The copy of the caller's arrays into the scene's planes (sg_create_scene,
sg_update_scene): every row width, Gaussian counts around a block of 128, and
arrays that start on a 16-byte boundary or 4 bytes past one.  The rendered
image must match the oracle's and not depend on the alignment."""
import numpy as np
import pytest

from tests import parity

pytestmark = pytest.mark.gpu


def _scene(n, degree):
    from paper_2510_12901_gb300 import synthetic as syn
    sc = syn.tiny_scene(seed=21, n=n)
    if degree is not None:
        rng = np.random.default_rng(22)
        sc.features = rng.normal(0.0, 0.3, (n, 3 * (degree + 1) ** 2)).astype(np.float32)
        sc.feature_kind, sc.sh_degree = syn.FEATURES_SH, degree
    # one Gaussian filling the middle of the view, so that the smallest scenes show
    sc.means[-1] = [0.0, -5.0, 0.0]
    sc.log_scales[-1] = [0.0, -0.5, 0.3]
    sc.opacity[-1] = 0.7
    return sc


def _device(a, shift):
    """A copy of `a` on the GPU that starts `shift` floats past a 16-byte boundary."""
    import torch
    buf = torch.empty(a.size + 4, dtype=torch.float32, device="cuda")
    t = buf[shift:shift + a.size]
    t.copy_(torch.from_numpy(np.ascontiguousarray(a).reshape(-1)))
    assert t.data_ptr() % 16 == 4 * shift
    return t.view(a.shape)


@pytest.mark.parametrize("degree", [None, 0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 1001])
def test_planes_of_every_width_and_alignment(n, degree):
    import torch
    from oracle import Oracle
    from paper_2510_12901_gb300 import simgut as sg, synthetic as syn
    sc, cam = _scene(n, degree), syn.tiny_camera()
    orc = Oracle(64).render_camera(sc, cam)
    C = sg.Camera(cam)
    outs = []
    for shift in (0, 1):
        S = sg.Scene(_scene(n, degree).subset(np.arange(n)[::-1]))    # other values first
        S.update(*[_device(getattr(sc, k), shift)
                   for k in ("means", "log_scales", "quats", "opacity", "features")])
        o = sg.render_camera(S, C, cam.c2w)
        torch.cuda.synchronize()
        outs.append([o[k].cpu().numpy() for k in ("rgb", "alpha", "depth")])
        rgb, alpha, depth = outs[-1]
        parity.compare_camera_rays(rgb.reshape(-1, 3), alpha.reshape(-1), depth.reshape(-1), orc,
                                   max_excluded=0.02, label=f"n={n} degree={degree}")
        assert alpha.max() > 0.1
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
