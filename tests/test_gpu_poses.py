"""Poses per row and per column where the projection takes another way to them:
row poses that are not 16-byte aligned (loaded 4 bytes at a time), and LiDARs
whose first column lies turns away from where azimuths are measured (columns
and culling cells wrap by the integer remainder)."""
import dataclasses

import numpy as np
import pytest

from paper_2510_12901_gb300 import synthetic as syn
from tests import parity as par

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", [0, 1])
def test_row_poses_off_a_16_byte_boundary(model):
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    cam = syn.street_cameras()[model]
    cam = dataclasses.replace(cam, width=210, height=131, fx=cam.fx / 9, fy=cam.fy / 9, cx=105.0,
                              cy=65.5)
    cam = syn.rolling_shutter(cam, speed=30.0, readout_s=0.05, yaw_rate=1.0)
    S, C = sg.Scene(syn.street_scene(20000, seed=71, length=60.0)), sg.Camera(cam)
    outs = []
    for shift in (0, 1, 2, 3):
        buf = torch.empty(cam.height * 12 + 4, device="cuda")
        rows = buf[shift:shift + cam.height * 12]
        rows.copy_(torch.from_numpy(cam.row_c2w).reshape(-1))
        assert rows.data_ptr() % 16 == 4 * shift
        o = sg.render_camera_rs(S, C, rows)
        torch.cuda.synchronize()
        outs.append([o[k].cpu().numpy() for k in ("rgb", "alpha", "depth")])
    assert outs[0][1].max() > 0.5
    for o in outs[1:]:
        for a, b in zip(outs[0], o):
            assert np.array_equal(a, b)


def _sweep(sc, L, keep):
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    fr = sg.Frame()
    sg.sg_frame_set_backward_state(fr.handle, keep)
    S, D = sg.Scene(sc), sg.Lidar(L)
    o = sg.render_lidar(S, D, L.col_c2w, frame=fr)
    torch.cuda.synchronize()
    return {k: o[k].cpu().numpy().reshape(-1) for k in ("range", "intensity", "drop", "alpha")}


@pytest.mark.parametrize("turns", [-3, -1, 1, 3])
@pytest.mark.parametrize("keep", [0, 1])
def test_first_column_turns_away(turns, keep):
    """The same columns named a few turns away: the same rays, up to the
    rounding of their azimuths (the oracle takes aliases one turn away only)."""
    sc = syn.street_scene(1500, seed=72, kind="lidar", length=60.0)
    L = syn.street_lidar(n_cols=256)          # columns 1.40625 degrees apart: exact azimuths
    a = _sweep(sc, L, keep)
    b = _sweep(sc, dataclasses.replace(L, az0_deg=L.az0_deg + 360.0 * turns), keep)
    hit = a["alpha"] > 0
    assert hit.sum() > 500
    for k in ("intensity", "drop", "alpha"):
        assert (np.abs(a[k] - b[k]) > par.TOL_ABS).mean() < 1e-3, k
    assert (np.abs(a["range"] - b["range"])[hit] > par.TOL_DEPTH_REL * a["range"][hit]).mean() < 1e-3
