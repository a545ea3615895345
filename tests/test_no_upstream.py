"""Autograd may run the backward of a render when none of its outputs has a
gradient: a later function that returns None for each is enough.  The parameters'
gradients are then 0, as with upstream gradients of zero, for both sensors."""
import types

import pytest
import torch

from paper_2510_12901_gb300 import autograd as sga
from paper_2510_12901_gb300 import synthetic as syn

SHAPES = [(7, 3), (7, 3), (7, 4), (7,), (7, 3)]


@pytest.mark.parametrize("fn,n_out", [(sga._RenderCamera, 3), (sga._RenderLidar, 4)])
def test_backward_without_any_gradient(fn, n_out):
    ctx = types.SimpleNamespace(shapes=[torch.Size(s) for s in SHAPES],
                                device=torch.device("cpu"), scene=None, frame=None)
    got = fn.backward(ctx, *[None] * n_out)
    assert len(got) == 10 and all(g is None for g in got[5:])
    assert [tuple(g.shape) for g in got[:5]] == SHAPES and not any(g.any() for g in got[:5])


class _Drop(torch.autograd.Function):
    """Uses its inputs and hands no gradient back."""

    @staticmethod
    def forward(ctx, *outs):
        return sum(o.sum() for o in outs)

    @staticmethod
    def backward(ctx, g):
        return (None,) * len(ctx.needs_input_grad)


@pytest.mark.gpu
@pytest.mark.parametrize("sensor", ["camera", "lidar"])
def test_render_whose_outputs_get_no_gradient(sensor):
    from paper_2510_12901_gb300 import simgut as sg
    if sensor == "camera":
        src, cam = syn.tiny_scene(n=300, seed=1), syn.tiny_camera()
        S, D, pose, render = sg.Scene(src), sg.Camera(cam), cam.c2w, sga.render_camera
    else:
        L = syn.street_lidar(n_cols=64)
        src = syn.street_scene(300, seed=1, kind="lidar", length=60.0)
        S, D, pose, render = sg.Scene(src), sg.Lidar(L), L.col_c2w, sga.render_lidar
    P = {k: torch.from_numpy(getattr(src, k)).float().cuda().requires_grad_()
         for k in sga._PARAMS}
    _Drop.apply(*render(P, S, D, pose)).backward()
    for p in P.values():
        assert p.grad.shape == p.shape and not p.grad.any()
