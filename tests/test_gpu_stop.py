"""A ray of the forward-only camera kernel that stops keeps T = -1 instead of a
flag.  Stopping thresholds from none (0: a ray never stops, T may reach 0) to a
third, alpha up to 1, lanes without a ray: the image must be the one of the
kernel that keeps the state of a backward, which has a flag."""
import dataclasses

import numpy as np
import pytest

from paper_2510_12901_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t_min", [0.0, 1e-4, 0.3])
@pytest.mark.parametrize("alpha_max", [0.99, 1.0])
@pytest.mark.parametrize("w,h", [(64, 64), (37, 21), (5, 3)])
def test_same_image_with_and_without_state(w, h, alpha_max, t_min):
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    sc = syn.layered_scene(seed=9, n=3000)      # several segments a tile
    sc.opacity[::7] = 1.0
    cam = dataclasses.replace(syn.tiny_camera(), width=w, height=h, cx=0.5 * w, cy=0.5 * h)
    opts = sg.sg_default_opts()
    opts.t_min, opts.alpha_max = t_min, alpha_max
    S, C, img = sg.Scene(sc), sg.Camera(cam), {}
    for keep in (0, 1):
        fr = sg.Frame()
        sg.sg_frame_set_backward_state(fr.handle, keep)
        o = sg.render_camera(S, C, cam.c2w, opts, frame=fr)
        torch.cuda.synchronize()
        img[keep] = torch.cat([o["rgb"].reshape(-1, 3), o["alpha"].reshape(-1, 1)], 1).cpu().numpy()
    assert img[1][:, 3].max() > 0.5
    # up to 3000 terms of at most 1, each rounded: 3000 2^-24 = 2e-4; a ray whose
    # alpha or T is within rounding of a threshold may differ by an entry (1%)
    e = np.abs(img[0].astype(np.float64) - img[1]).max(axis=1)
    assert np.isfinite(img[0]).all() and (e > 2e-4).mean() <= 0.01, e.max()
