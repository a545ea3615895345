"""The one-block depth stage of small scenes at the sizes where its warps' runs
of 32 and 128 entries end, and past its largest (4096): the pair lists of
test_gpu_sort, and a frame whose scratch a larger scene has grown before."""
import numpy as np
import pytest

from tests.test_gpu_sort import test_pair_list_order as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 31, 32, 33, 127, 128, 129, 1000, 1025, 4095, 4098])
@pytest.mark.parametrize("ties", [False, True])
def test_small_scene(n, ties):
    check(n, ties, 64, 64)


def test_after_a_larger_scene():
    import dataclasses
    import torch
    from paper_2510_12901_gb300 import simgut as sg, synthetic as syn
    cam = dataclasses.replace(syn.tiny_camera(), width=512, height=512, fx=480.0, fy=480.0, cx=256.0,
                              cy=256.0)
    big, small = (sg.Scene(syn.tiny_scene(seed=7, n=n)) for n in (60000, 4000))
    C, fr = sg.Camera(cam), sg.Frame()
    want = sg.render_camera(small, C, cam.c2w, frame=sg.Frame())["rgb"].cpu().numpy()
    for S in (big, small, big, small, small):
        o = sg.render_camera(S, C, cam.c2w, frame=fr)
        torch.cuda.synchronize()
        sg.sg_frame_status(fr.handle)
        if S is small:
            assert np.array_equal(o["rgb"].cpu().numpy(), want)
