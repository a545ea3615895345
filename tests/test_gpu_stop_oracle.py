"""Stopping rays at thresholds from none (0: a ray never stops, T may reach 0) to a
third, with alpha up to 1, against the 64-bit oracle: colour, alpha and depth of the
camera, range, intensity, drop and alpha of the LiDAR, through the kernels that keep
the state of a backward and those that do not.  They mark a stopped ray in T itself
(T = -1, -T or 0), which at t_min = 0 or alpha = 1 comes closest to a live ray's T."""
import dataclasses

import numpy as np
import pytest

from paper_2510_12901_gb300 import synthetic as syn
from tests import parity as par

pytestmark = pytest.mark.gpu
OPTS = [(t, a) for t in (0.0, 1e-4, 0.3) for a in (0.99, 1.0)]


def _unsure(orc, t_min):
    # near alpha = 1 the stop test compares T (1 - alpha), whose error is that of
    # alpha, 2e-6, times T <= 1: relative to t_min this passes the common margin
    return orc["m_tmin"] < 2e-6 / t_min if t_min > 0 else np.zeros(len(orc), bool)


@pytest.mark.parametrize("keep", [0, 1])
@pytest.mark.parametrize("t_min,alpha_max", OPTS)
@pytest.mark.parametrize("w,h", [(64, 64), (37, 21)])
def test_camera(O64, w, h, t_min, alpha_max, keep):
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    sc = syn.layered_scene(seed=9, n=3000)      # several segments a tile
    sc.opacity[::7] = 1.0
    cam = dataclasses.replace(syn.tiny_camera(), width=w, height=h, cx=0.5 * w, cy=0.5 * h)
    fr = sg.Frame()
    sg.sg_frame_set_backward_state(fr.handle, keep)
    o = sg.render_camera(sg.Scene(sc), sg.Camera(cam), cam.c2w,
                         sg.sg_default_opts(t_min=t_min, alpha_max=alpha_max), frame=fr)
    torch.cuda.synchronize()
    orc = O64.render_camera(sc, cam, O64.opts(t_min=t_min, alpha_max=alpha_max))
    assert orc["alpha"].max() > (0.5 if t_min > 0.1 else 0.99)
    # the common margins exclude at most what they may in the other layered scene; a
    # tenth of the rays cross T = 1e-4 within 2% of it
    unsure = _unsure(orc, t_min)
    assert unsure.mean() < 0.12
    par.compare_camera_rays(o["rgb"].cpu().numpy().reshape(-1, 3),
                            o["alpha"].cpu().numpy().reshape(-1),
                            o["depth"].cpu().numpy().reshape(-1), orc,
                            max_excluded=0.07 + unsure.mean(), also_excluded=unsure)


@pytest.mark.parametrize("keep", [0, 1])
@pytest.mark.parametrize("t_min,alpha_max", OPTS)
def test_lidar(O64, t_min, alpha_max, keep):
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    L = syn.street_lidar(n_cols=128)
    sc = syn.street_scene(1500, seed=10, kind="lidar", length=60.0)
    sc.log_scales += 0.7                        # lists of several segments near the sensor
    sc.opacity[::7] = 1.0
    fr = sg.Frame()
    sg.sg_frame_set_backward_state(fr.handle, keep)
    o = sg.render_lidar(sg.Scene(sc), sg.Lidar(L), L.col_c2w,
                        sg.sg_default_opts(t_min=t_min, alpha_max=alpha_max), frame=fr)
    torch.cuda.synchronize()
    orc = O64.render_lidar(sc, L, O64.opts(t_min=t_min, alpha_max=alpha_max))
    assert (orc["n_contrib"] > 0).sum() > 1000
    par.compare_lidar_rays(*[o[k].cpu().numpy().reshape(-1)
                             for k in ("range", "intensity", "drop", "alpha")], orc,
                           also_excluded=_unsure(orc, t_min))
