"""The compositing's work items at the tile counts where their kernels' shares
end (256 tiles a block, 12288 for the one-launch form): an image cropped to
fewer tiles, with the same intrinsics, shows the same pixels bit for bit."""
import dataclasses

import pytest

pytestmark = pytest.mark.gpu
FULL = (2000, 2048)        # 125 x 128 = 16000 tiles: the two grid-wide kernels


@pytest.fixture(scope="module")
def full():
    import numpy as np
    from paper_2510_12901_gb300 import simgut as sg, synthetic as syn
    sc = syn.tiny_scene(seed=61, n=4000)
    sc.means[:, 1] = np.random.default_rng(62).uniform(-8.0, 10.0, sc.n)
    # a crowd whose tiles' lists are split, in the corner every crop shows
    sc.means[:1200] = np.random.default_rng(63).uniform(-0.5, 0.5, (1200, 3)) * [0.2, 1.0, 0.2] + \
        [-9.5, 0.0, 9.5]
    cam = dataclasses.replace(syn.tiny_camera(), width=FULL[0], height=FULL[1], fx=900.0, fy=900.0,
                              cx=1000.0, cy=1020.0)
    S = sg.Scene(sc)
    return S, cam, {keep: _render(sg, S, cam, keep) for keep in (0, 1)}


def _render(sg, S, cam, keep):
    import torch
    fr, C = sg.Frame(), sg.Camera(cam)
    sg.sg_frame_set_backward_state(fr.handle, keep)
    o = sg.render_camera(S, C, cam.c2w, frame=fr)
    torch.cuda.synchronize()
    return {k: o[k] for k in ("rgb", "alpha", "depth")}


@pytest.mark.parametrize("tx,ty", [(1, 1), (51, 5), (64, 4), (86, 3), (93, 11), (64, 16), (41, 25),
                                   (96, 128), (110, 112)])
@pytest.mark.parametrize("keep", [0, 1])
def test_crop_shows_the_same_pixels(full, tx, ty, keep):
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    S, cam, ref = full
    w, h = 16 * tx, 16 * ty
    out = _render(sg, S, dataclasses.replace(cam, width=w, height=h), keep)
    assert float(ref[keep]["alpha"].max()) > 0.5
    for k, v in out.items():
        assert torch.equal(v, ref[keep][k][:h, :w]), k
