"""Capacity mode with 2^32 pairs and more in view: the pairs beyond the capacity are
dropped, the nearest Gaussians' pairs are kept in order, and nothing is read or
written out of range (offsets beyond 32 bits must not wrap into the kept ones)."""
import dataclasses

import numpy as np
import pytest

from paper_2510_12901_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def test_capacity_far_below_the_pairs_in_view():
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    # 70000 opaque sheets across a view of 65536 tiles: 4.6e9 pairs, 8M kept.  The
    # table of first owners ends at some 5M pairs, the blocks after it search.
    n, side, cap = 70000, 4096, 8000000
    rng = np.random.default_rng(61)
    sc = syn.tiny_scene(seed=60, n=n)
    sc.means[:] = 0.0
    sc.means[:, 1] = rng.permutation(np.linspace(0.0, 7.0, n))
    sc.log_scales[:] = np.log([50.0, 0.01, 50.0])
    sc.quats[:] = [1.0, 0.0, 0.0, 0.0]
    sc.opacity[:] = 0.9
    cam = dataclasses.replace(syn.tiny_camera(), width=side, height=side, fx=4000.0, fy=4000.0,
                              cx=side / 2, cy=side / 2)
    C = sg.Camera(cam)
    # a ray stops after four entries of alpha 0.9 (T < 1e-4 at the fifth), so the
    # nearest 50 Gaussians alone give the same image, bit for bit
    near = sc.subset(np.sort(np.argsort(sc.means[:, 1])[:50]))
    S, fr = sg.Scene(near), sg.Frame()
    want = sg.render_camera(S, C, cam.c2w, frame=fr)
    torch.cuda.synchronize()
    assert fr.stats()[0] == 50 * 65536 and float(want["alpha"].min()) > 0.999
    S, fr = sg.Scene(sc), sg.Frame()
    sg.sg_frame_set_capacity(fr.handle, cap)
    got = sg.render_camera(S, C, cam.c2w, frame=fr)
    torch.cuda.synchronize()
    sg.sg_frame_status(fr.handle)
    assert sg.sg_frame_dropped_pairs(fr.handle) == (0xffffffff - cap, cap)
    ids = fr.field(sg.FIELD_PAIR_IDS, np.uint32).reshape(-1)
    order = np.argsort(sc.means[:, 1])
    assert np.array_equal(np.unique(ids), np.sort(order[:(cap + 65535) // 65536]))
    for k in ("rgb", "alpha", "depth"):
        assert torch.equal(got[k], want[k]), k
