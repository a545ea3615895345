"""The depth sort, pair offsets, binning and tile sort at the sizes where their
tiles and look-back rounds end: the pair list must be the Gaussians' pairs in
(tile, depth, id) order, from the projection's own keys and tile ranges."""
import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _expected(tiles, depth, count, ntx):
    """(tile, id) of every pair in (tile, depth, id) order."""
    ids = np.nonzero(count)[0]
    ids = ids[np.argsort(depth[ids], kind="stable")]
    t = tiles[ids]
    w = t[:, 1] - t[:, 0] + 1
    n = w * (t[:, 3] - t[:, 2] + 1)
    assert np.array_equal(n, count[ids])
    owner = np.repeat(np.arange(len(ids)), n)
    local = np.arange(n.sum()) - np.repeat(np.cumsum(n) - n, n)
    tile = (t[owner, 2] + local // w[owner]) * ntx + t[owner, 0] + local % w[owner]
    order = np.argsort(tile, kind="stable")
    return tile[order].astype(np.uint32), ids[owner][order].astype(np.uint32)


# tiles of 2048 (compaction, offsets up to 262144 Gaussians), 4096 (radix passes)
# and 8192 (offsets above) entries;
# 32 of them a look-back round
@pytest.mark.parametrize("n", [1, 2, 2047, 2049, 4096, 4097, 8193, 66000, 135000, 262144,
                               300001])
@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("w,h", [(16, 16), (64, 64), (1030, 517)])
def test_pair_list_order(n, ties, w, h):
    import torch
    from paper_2510_12901_gb300 import simgut as sg, synthetic as syn
    sc = syn.tiny_scene(seed=41, n=n)
    rng = np.random.default_rng(42)
    sc.means[:, 1] = rng.uniform(-8.0, 10.0, n)      # most of them in view
    sc.means[:, [0, 2]] *= 0.05 * (sc.means[:, 1:2] + 10.0)
    if n > 100000:
        sc.log_scales -= 1.0
    if ties:                        # runs of Gaussians at one place: equal keys, id order
        sc.means[:] = sc.means[(np.arange(n) // 3) * 3]
    f = 60.0 * w / 64.0
    cam = dataclasses.replace(syn.tiny_camera(), width=w, height=h, fx=f, fy=f, cx=w / 2, cy=h / 2)
    S, C, fr = sg.Scene(sc), sg.Camera(cam), sg.Frame()
    for _ in range(2):              # the second render reuses the workspace
        sg.render_camera(S, C, cam.c2w, frame=fr)
    torch.cuda.synchronize()
    sg.sg_frame_status(fr.handle)
    tiles = fr.field(sg.FIELD_TILES, np.int32, 4)
    depth, count = fr.field(sg.FIELD_DEPTH, np.float32), fr.field(sg.FIELD_COUNT, np.uint32)
    ntx = (w + 15) // 16
    tile, ids = _expected(tiles, depth, count, ntx)
    assert np.array_equal(fr.field(sg.FIELD_PAIR_TILES, np.uint32), tile)
    assert np.array_equal(fr.field(sg.FIELD_PAIR_IDS, np.uint32), ids)
    r = fr.field(sg.FIELD_RANGES, np.uint32, 2)
    per = np.bincount(tile, minlength=len(r))
    assert np.array_equal(r[:, 1] - r[:, 0], per)
    assert np.array_equal(r[per > 0, 0], (np.cumsum(per) - per)[per > 0])


def test_more_pairs_than_the_owner_table():
    """A few Gaussians over every tile of a large image: binning blocks beyond
    the table of first owners search the offsets for theirs."""
    import torch
    from paper_2510_12901_gb300 import simgut as sg, synthetic as syn
    n = 403
    sc = syn.tiny_scene(seed=43, n=n)
    sc.means[:] = np.random.default_rng(44).uniform(-0.5, 0.5, (n, 3)) + [0.0, 8.0, 0.0]
    sc.log_scales[:] = np.log(4.0)
    cam = dataclasses.replace(syn.tiny_camera(), width=2000, height=2041, fx=900.0, fy=900.0,
                              cx=1000.0, cy=1020.0)
    S, C, fr = sg.Scene(sc), sg.Camera(cam), sg.Frame()
    sg.sg_frame_set_backward_state(fr.handle, 0)
    sg.render_camera(S, C, cam.c2w, frame=fr)
    torch.cuda.synchronize()
    sg.sg_frame_status(fr.handle)
    tile, ids = _expected(fr.field(sg.FIELD_TILES, np.int32, 4),
                          fr.field(sg.FIELD_DEPTH, np.float32),
                          fr.field(sg.FIELD_COUNT, np.uint32), 125)
    assert len(ids) > 2048 * (n // 64 + 1024)
    assert np.array_equal(fr.field(sg.FIELD_PAIR_TILES, np.uint32), tile)
    assert np.array_equal(fr.field(sg.FIELD_PAIR_IDS, np.uint32), ids)
