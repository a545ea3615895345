"""The rolling-shutter and LiDAR compositing queue the list entries that reach
a ray and stage them 32 at a time.  Lists of every remainder around one, two
and three stages, every third entry a small one that few sub-blocks see: each
ray must match the oracle, which walks the list entry by entry."""
import dataclasses

import numpy as np
import pytest

from paper_2510_12901_gb300 import synthetic as syn
from tests import parity as par

pytestmark = pytest.mark.gpu
COUNTS = [1, 31, 32, 33, 63, 64, 65, 97]


def _ahead(sc, n, eye, right, ahead, up, seed):
    """The scene's n Gaussians as translucent layers around the direction
    `ahead` from `eye`, their depths well apart."""
    rng = np.random.default_rng(seed)
    r = 4.0 + 20.0 * (rng.permutation(n) + 0.5) / n
    s = np.where(np.arange(n) % 3 == 2, 0.01, 0.15) * r
    uv = rng.uniform(-0.05, 0.05, (n, 2))
    d = ahead + uv[:, :1] * right + uv[:, 1:] * up
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    sc.means[:] = eye + d * r[:, None]
    sc.log_scales[:] = np.log(s)[:, None] + rng.uniform(-0.2, 0.2, (n, 3))
    sc.opacity[:] = rng.uniform(0.02, 0.06, n)
    return sc


@pytest.mark.parametrize("n", COUNTS)
def test_rolling_shutter(O64, n):
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    cam = dataclasses.replace(syn.tiny_camera(), width=17, height=14, fx=60.0, fy=60.0, cx=8.5,
                              cy=7.0)
    cam = syn.rolling_shutter(cam, speed=2.0)
    M = np.asarray(cam.c2w, np.float64).reshape(3, 4)
    R, eye = M[:, :3], M[:, 3]
    sc = _ahead(syn.tiny_scene(seed=n, n=n), n, eye, R[:, 0], R[:, 2], R[:, 1], seed=n)
    S, C = sg.Scene(sc), sg.Camera(cam)
    o = sg.render_camera_rs(S, C, cam.row_c2w)
    torch.cuda.synchronize()
    orc = O64.render_camera(sc, cam)
    # rays at a small Gaussian's rim may be ambiguous: a tenth at most
    par.compare_camera_rays(o["rgb"].cpu().numpy().reshape(-1, 3),
                            o["alpha"].cpu().numpy().reshape(-1),
                            o["depth"].cpu().numpy().reshape(-1), orc, max_excluded=0.1,
                            label=f"rolling shutter, {n} entries", posed=True)


@pytest.mark.parametrize("mode", ["saved", "forward"])
@pytest.mark.parametrize("n", COUNTS)
def test_lidar(O64, n, mode):
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    L = syn.street_lidar(n_beams=64, n_cols=128)
    eye = np.asarray(L.col_c2w, np.float64).reshape(-1, 3, 4)[64, :, 3]
    sc = syn.street_scene(n, seed=n, kind="lidar", length=60.0)
    sc = _ahead(sc, n, eye, *np.eye(3), seed=n)
    S, Ld, fr = sg.Scene(sc), sg.Lidar(L), sg.Frame()
    sg.sg_frame_set_backward_state(fr.handle, 1 if mode == "saved" else 0)
    o = sg.render_lidar(S, Ld, L.col_c2w, None, frame=fr)
    torch.cuda.synchronize()
    g = {k: o[k].cpu().numpy().reshape(-1) for k in ("range", "intensity", "drop", "alpha")}
    orc = O64.render_lidar(sc, L)
    assert (orc["alpha"] > 0).any()
    par.compare_lidar_rays(g["range"], g["intensity"], g["drop"], g["alpha"], orc,
                           max_excluded=0.1, label=f"lidar {mode}, {n} entries")
