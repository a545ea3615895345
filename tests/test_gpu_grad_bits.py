"""dL/dsigma and dL/dalpha to the last bit, where the arithmetic of one or two entries
a ray leaves nothing to the order of sums: dL/dsigma is dL/dalpha rho, without a
division, and the remainder of a ray is divided by 1 - alpha as IEEE 754 rounds it.
One-pose cameras and rolling shutters (whose walk the LiDAR shares)."""
import dataclasses

import numpy as np
import pytest

from paper_2510_12901_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu
SIDE, STEP = 64, 2          # Gaussians sit on every second pixel of a 64x64 image


def _dots(depth, opacity, feature, rng):
    """Gaussians of 0.2 pixels, one ray each: the next pixel is at least 3.5 of their
    standard deviations away (alpha < 0.0022, below alpha_min = 1/255)."""
    px = np.arange(0, SIDE, STEP) + 0.5
    u, v = [a.reshape(-1) for a in np.meshgrid(px, px)]
    n = len(u)
    u, v = u + rng.uniform(-0.25, 0.25, n), v + rng.uniform(-0.25, 0.25, n)
    sc = syn.tiny_scene(seed=71, n=n)
    z = depth * np.ones(n)
    sc.means[:] = np.stack([(u - 32.0) / 60.0 * z, z - 10.0, -(v - 32.0) / 60.0 * z], 1)
    sc.log_scales[:] = np.log(0.2 / 60.0 * depth)
    sc.opacity[:] = opacity
    sc.features[:] = feature
    return sc


def _grads(sc, rolling):
    """Gradients of the sum of the first channel, and that channel."""
    import torch
    from paper_2510_12901_gb300 import simgut as sg
    cam = syn.tiny_camera()
    S, C, fr = sg.Scene(sc), sg.Camera(cam), sg.Frame()
    if rolling:
        rows = np.tile(np.asarray(cam.c2w, np.float32).reshape(1, 12), (SIDE, 1))
        o = sg.render_camera_rs(S, C, torch.from_numpy(rows).cuda(), frame=fr)
    else:
        o = sg.render_camera(S, C, cam.c2w, frame=fr)
    up = torch.zeros_like(o["rgb"])
    up[..., 0] = 1.0
    n = sc.n
    g = [torch.full(s, float("nan"), device="cuda") for s in ((n, 3), (n, 3), (n, 4), (n,), (n, 3))]
    sg.sg_backward_camera_write(S.handle, fr.handle, up.data_ptr(), 0, 0,
                                sg.sg_grads(*[x.data_ptr() for x in g]),
                                torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return g[3].cpu().numpy(), g[4].cpu().numpy()[:, 0], o["rgb"].cpu().numpy()[..., 0]


@pytest.mark.parametrize("rolling", [False, True])
def test_one_entry_a_ray(rolling):
    # one feature of 1: dL/dalpha = 1, so dL/dsigma = rho and dL/dfeature = alpha = sigma rho
    rng = np.random.default_rng(72)
    sc = _dots(5.0, rng.uniform(0.1, 0.95, (SIDE // STEP) ** 2), 1.0, rng)
    g_sigma, g_feat, img = _grads(sc, rolling)
    # no ray has another Gaussian's entry; rho is at least exp(-1.25^2) = 0.2096
    assert not img[1::STEP].any() and not img[:, 1::STEP].any()
    assert np.array_equal(img[::STEP, ::STEP].reshape(-1), g_feat) and g_sigma.min() > 0.2
    assert np.array_equal(sc.opacity * g_sigma, g_feat)


@pytest.mark.parametrize("rolling", [False, True])
def test_two_entries_a_ray(rolling):
    # a front entry of feature 0 and sigma 1/2, one behind it of feature 1: with F the
    # ray's sum, dL/dalpha = -F / (1 - alpha) and rho = 2 alpha of the front entry
    rng = np.random.default_rng(73)
    m = (SIDE // STEP) ** 2
    a = _dots(5.0, 0.5, 0.0, rng)
    b = _dots(6.0, rng.uniform(0.3, 0.95, m), 1.0, rng)
    sc = dataclasses.replace(a, **{k: np.concatenate([getattr(a, k), getattr(b, k)])
                                   for k in ("means", "log_scales", "quats", "opacity", "features")})
    g_sigma, g_feat, img = _grads(sc, rolling)
    F = img[::STEP, ::STEP].reshape(-1)
    alpha = g_feat[:m]
    # at least 0.3 0.2096 (1 - 0.5) and 0.5 0.2096
    assert F.min() > 0.03 and alpha.min() > 0.1
    one = np.float32(1.0)
    want = -(F / (one - alpha)) * (np.float32(2.0) * alpha)
    assert want.dtype == np.float32 and np.array_equal(g_sigma[:m], want)
