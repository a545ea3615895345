"""The work this renderer is timed on: its public entry points over the sizes its
users call them with.

A case is a dict of plain values; `kind` names the call it stands for:

  camera        one view through render_camera / render_camera_rs
  rig           a vehicle's fisheye and pinhole views in one sg_render_cameras call
  static        one small view through the allocation-free sg_render_camera_static
  lidar         one spinning-LiDAR sweep through render_lidar
  train_camera  scene update, camera render and backward through the autograd wrapper
  train_lidar   the same for a LiDAR sweep
  serve         a burst of mixed requests through the request server

Scenes follow the repository's synthetic inputs (the 20 m cube and the street of
surface-aligned Gaussians), drawn on the GPU from the seed; sensors are those of
`paper_2510_12901_gb300.synthetic`.  `exact` evaluates the renderer's definition in
64 bits over (ray, Gaussian) pairs with torch alone, without tiles.
"""
import dataclasses
import math
import types

import numpy as np
import torch

from paper_2510_12901_gb300 import autograd as sga
from paper_2510_12901_gb300 import simgut as sg
from paper_2510_12901_gb300 import synthetic as syn
from paper_2510_12901_gb300.serve import Server

PARAMS = ("means", "log_scales", "quats", "opacity", "features")


# ----------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: 4096 RGB Gaussians into 64x64, launches and latency count
        dict(name="tiny_camera", kind="camera", scene="cube", n=4096, model="pinhole",
             width=64, height=64, degree=0, state=True, rolling=False, actors=0),
        # the deployment variant that allocates nothing, near its pair limit, odd image
        dict(name="static_251x243", kind="static", scene="cube", n=20011, model="pinhole",
             width=251, height=243, degree=0),
        # a ragged inference view of a street tile with moving cars
        dict(name="fisheye_641x479_actors", kind="camera", scene="street", n=150001,
             model="fisheye", width=641, height=479, degree=1, state=False, rolling=False,
             actors=16),
        # the flagship frame: both street cameras of 1M Gaussians, degree-3 SH
        dict(name="rig_1m", kind="rig", scene="street", n=1000000, degree=3, rolling=False),
        # one request's view of a large resident scene
        dict(name="pinhole_1080p_2m", kind="camera", scene="street", n=2000000,
             model="pinhole", width=1920, height=1080, degree=3, state=False, rolling=False,
             actors=0),
        # a rolling-shutter camera: a pose per pixel row
        dict(name="rolling_fisheye_1m", kind="camera", scene="street", n=1000000,
             model="fisheye", width=1920, height=1280, degree=3, state=False, rolling=True,
             actors=0),
        # the flagship LiDAR sweep: 128 beams x 2048 columns, 2M Gaussians, moving sensor
        dict(name="lidar_128x2048_2m", kind="lidar", n=2000000, beams=128, cols=2048, sh=False,
             degree=0, beam_mrad=0.0, state=False),
        # a smaller LiDAR with view-dependent features and beam divergence
        dict(name="lidar_64x1024_sh_beam", kind="lidar", n=500000, beams=64, cols=1024, sh=True,
             degree=3, beam_mrad=3.0, state=False),
        # one differentiable camera step at full size
        dict(name="train_fisheye_1m", kind="train_camera", scene="street", n=1000000,
             model="fisheye", width=1920, height=1280, degree=3),
        # a fitting loop on a small crop, odd sizes
        dict(name="train_crop_333x251", kind="train_camera", scene="street", n=40009,
             model="pinhole", width=333, height=251, degree=2),
        # one differentiable LiDAR step at full size
        dict(name="train_lidar_2m", kind="train_lidar", n=2000000, beams=128, cols=2048,
             sh=False, degree=0),
        # twelve waiting requests, three of each sensor of the serving mix
        dict(name="serve_12_requests", kind="serve", n=500000, requests=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("camera", "camera", "camera", "rig", "static", "lidar", "lidar",
                       "train_camera", "train_camera", "train_lidar", "serve"))
    if kind == "rig":
        return dict(kind=kind, scene="street", n=_log_int(rng, 100000, 1000000),
                    degree=rng.randint(0, 3), rolling=rng.random() < 0.3)
    if kind == "static":
        w = rng.randint(64, 255)
        return dict(kind=kind, scene="cube", n=_log_int(rng, 1000, 20000), model="pinhole",
                    width=w, height=rng.randint(64, 255), degree=0)
    if kind == "lidar":
        return dict(kind=kind, n=_log_int(rng, 50000, 2000000), beams=rng.choice((64, 128)),
                    cols=rng.choice((512, 1024, 1800, 2048)), sh=rng.random() < 0.5,
                    degree=rng.randint(0, 3), beam_mrad=rng.choice((0.0, 0.0, 3.0)),
                    state=rng.random() < 0.3)
    if kind == "train_lidar":
        return dict(kind=kind, n=_log_int(rng, 20000, 2000000), beams=rng.choice((64, 128)),
                    cols=rng.choice((256, 512, 1024, 2048)), sh=rng.random() < 0.3,
                    degree=rng.randint(0, 3))
    if kind == "serve":
        return dict(kind=kind, n=_log_int(rng, 100000, 600000), requests=rng.randint(2, 12))
    width = _log_int(rng, 64, 1920)
    height = max(48, min(1280, int(width * rng.uniform(0.5, 0.8))))
    case = dict(kind=kind, scene="street", n=_log_int(rng, 4096, 1000000),
                model=rng.choice(("pinhole", "fisheye")), width=width, height=height,
                degree=rng.randint(0, 3))
    if kind == "camera":
        rolling = rng.random() < 0.25
        case.update(state=rng.random() < 0.3, rolling=rolling,
                    actors=rng.choice((0, 0, 16)))
    return case


# -------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1000003 * (seed % 1000003) + 17)


def _unit_quats(g, n):
    q = torch.randn((n, 4), generator=g, device="cuda")
    return q / q.norm(dim=1, keepdim=True)


def _cube(n, seed):
    """Gaussians in a 20 m cube (`synthetic.tiny_scene`)."""
    g = _gen(seed)

    def u(*s):
        return torch.rand(s, generator=g, device="cuda")

    return types.SimpleNamespace(
        means=20.0 * u(n, 3) - 10.0,
        log_scales=-1.5 + 0.5 * torch.randn((n, 3), generator=g, device="cuda"),
        quats=_unit_quats(g, n),
        opacity=torch.sigmoid(torch.randn(n, generator=g, device="cuda")),
        features=u(n, 3), feature_kind=syn.FEATURES_RGB, sh_degree=0, actor_of=None,
        actor_poses=None)


def _street(n, seed, kind, degree=0, actors=0):
    """The street of `synthetic.street_scene`: 45% ground, 45% facades, 10% clutter over
    150 m, flattened along the surface normal; `actors`: a tenth of the Gaussians on that
    many cars (`synthetic.with_actors`)."""
    g = _gen(seed)

    def u(m, lo, hi):
        return lo + (hi - lo) * torch.rand(m, generator=g, device="cuda")

    def randn(*s):
        return torch.randn(s, generator=g, device="cuda")

    ng = nf = int(round(0.45 * n))
    nc = n - ng - nf
    side = torch.where(u(nf, 0.0, 1.0) < 0.5, -12.0, 12.0)
    means = torch.cat([
        torch.stack([u(ng, 0.0, 150.0), u(ng, -10.0, 10.0), torch.zeros(ng, device="cuda")], 1),
        torch.stack([u(nf, 0.0, 150.0), side, u(nf, 0.0, 15.0)], 1),
        torch.stack([u(nc, 0.0, 150.0), u(nc, -12.0, 12.0), u(nc, 0.0, 15.0)], 1)])
    means = means + 0.05 * randn(n, 3)
    # the surface's quaternion times a small rotation (clutter: any rotation)
    axis = randn(n, 3)
    axis = axis / axis.norm(dim=1, keepdim=True)
    half = 0.05 * randn(n)
    w, v = torch.cos(half), axis * torch.sin(half)[:, None]
    c = math.cos(math.pi / 4)
    qf = torch.stack([c * w - c * v[:, 0], c * v[:, 0] + c * w, c * v[:, 1] - c * v[:, 2],
                      c * v[:, 2] + c * v[:, 1]], 1)
    quats = torch.cat([w[:, None], v], 1)
    quats[ng:ng + nf] = qf[ng:ng + nf]
    quats[ng + nf:] = _unit_quats(g, nc)
    log_scales = math.log(0.05) + 0.5 * randn(n, 3)
    log_scales[:ng + nf, 2] += math.log(0.2)
    if kind == "camera":
        opacity = torch.sigmoid(randn(n))
        features = 0.3 * randn(n, 3 * (degree + 1) ** 2)
        fk = syn.FEATURES_SH
    else:
        opacity = torch.sigmoid(torch.where(u(n, 0.0, 1.0) < 0.7, 4.0, -4.0) + randn(n))
        features = torch.cat([u(n, 0.0, 1.0)[:, None], randn(n, 2)], 1)
        fk = syn.FEATURES_LIDAR
        if kind == "lidar_sh":
            sh = 0.3 * randn(n, (degree + 1) ** 2, 3)
            sh[:, 0, :] = 3.5 * features
            features, fk = sh.reshape(n, -1).contiguous(), syn.FEATURES_LIDAR_SH
    sc = types.SimpleNamespace(means=means, log_scales=log_scales, quats=quats,
                               opacity=opacity, features=features, feature_kind=fk,
                               sh_degree=degree if fk != syn.FEATURES_LIDAR else 0,
                               actor_of=None, actor_poses=None)
    if actors:
        on = u(n, 0.0, 1.0) < 0.1
        who = torch.randint(0, actors, (n,), generator=g, device="cuda", dtype=torch.int32)
        half = torch.tensor([2.25, 0.9, 0.75], device="cuda")
        face = torch.randint(0, 3, (n, 1), generator=g, device="cuda")
        local = (2.0 * torch.rand((n, 3), generator=g, device="cuda") - 1.0) * half
        pick = torch.zeros_like(local, dtype=torch.bool).scatter_(1, face, True)
        local = torch.where(pick, torch.where(local < 0, -half, half), local)
        local[:, 2] += 0.75
        sc.means = torch.where(on[:, None], local, sc.means).contiguous()
        sc.actor_of = torch.where(on, who, -1).cpu().numpy()
        rng = np.random.default_rng(seed)
        sc.actor_poses = np.stack([
            syn.actor_pose(rng.uniform(5.0, 140.0), rng.choice([-1.0, 1.0]) * rng.uniform(1.5, 6.0),
                           rng.uniform(-math.pi, math.pi)) for _ in range(actors)])
    return sc


def _look(rng, cam):
    """`cam` near the start of the street, looking down it."""
    yaw = rng.uniform(-0.1, 0.1)
    c2w = syn._look_c2w([rng.uniform(0.0, 15.0), rng.uniform(-3.0, 3.0), 1.6],
                        [math.cos(yaw), math.sin(yaw), 0.0], [0.0, 0.0, -1.0])
    return dataclasses.replace(cam, c2w=c2w)


def _camera(case, seed):
    """The case's sensor: the street cameras scaled to the image, or the cube's camera."""
    rng = np.random.default_rng(seed)
    w, h = case["width"], case["height"]
    if case["scene"] == "cube":
        f = 60.0 * max(w, h) / 64.0
        return dataclasses.replace(syn.tiny_camera(), width=w, height=h, fx=f, fy=f,
                                   cx=0.5 * w, cy=0.5 * h)
    fish, pin = syn.street_cameras(seed=seed)
    base = fish if case["model"] == "fisheye" else pin
    s = w / base.width
    cam = dataclasses.replace(base, width=w, height=h, fx=base.fx * s, fy=base.fy * s,
                              cx=0.5 * w, cy=0.5 * h)
    cam = _look(rng, cam)
    return syn.rolling_shutter(cam) if case.get("rolling") else cam


def _rig_cameras(case, seed):
    rng = np.random.default_rng(seed)
    cams = [_look(rng, c) for c in syn.street_cameras(seed=seed)]
    cams[1] = dataclasses.replace(cams[1], c2w=cams[0].c2w)    # one vehicle
    return [syn.rolling_shutter(c) for c in cams] if case["rolling"] else cams


def _lidar(case, seed):
    rng = np.random.default_rng(seed)
    L = syn.street_lidar(n_beams=case["beams"], n_cols=case["cols"])
    start = (rng.uniform(20.0, 60.0), rng.uniform(-3.0, 3.0), 1.8)
    return dataclasses.replace(L, col_c2w=syn.sweep_poses(
        L.n_cols, start, yaw0=rng.uniform(-math.pi, math.pi)))


def _scene(case, seed):
    if case["kind"] in ("lidar", "train_lidar"):
        return _street(case["n"], seed, "lidar_sh" if case["sh"] else "lidar", case["degree"])
    if case["scene"] == "cube":
        return _cube(case["n"], seed)
    return _street(case["n"], seed, "camera", case["degree"], case.get("actors", 0))


def _upstream(shapes, seed):
    """What a mean loss over the rays hands back, per output."""
    g = _gen(seed + 7)
    return {k: torch.randn(s, generator=g, device="cuda") / float(s[0] * s[1])
            for k, s in shapes.items()}


def _image(h, w):
    return [torch.empty((h, w, 3), device="cuda"), torch.empty((h, w), device="cuda"),
            torch.empty((h, w), device="cuda")]


def _frame(state):
    fr = sg.Frame()
    sg.sg_frame_set_backward_state(fr.handle, state)
    return fr


def _serve_parts(case, seed):
    """The serving mix: one camera scene (two thirds of the Gaussians) and one LiDAR
    scene, and (sensor, pose) of each request in arrival order."""
    rng = np.random.default_rng(seed)
    n_cam = 2 * case["n"] // 3
    scenes = dict(camera=_street(n_cam, seed, "camera", 3),
                  lidar=_street(case["n"] - n_cam, seed + 1, "lidar"))
    fish, pin = syn.street_cameras(seed=seed)
    fish = dataclasses.replace(fish, width=1280, height=960, cx=640.0, cy=480.0)
    sensors = [pin, fish, syn.street_lidar(64, 1024), syn.street_lidar(128, 2048)]
    reqs = []
    for i in range(case["requests"]):
        s = sensors[i % 4]
        if isinstance(s, syn.Camera):
            reqs.append((i % 4, _look(rng, s)))
        else:
            start = (rng.uniform(20.0, 60.0), rng.uniform(-3.0, 3.0), 1.8)
            reqs.append((i % 4, dataclasses.replace(s, col_c2w=syn.sweep_poses(
                s.n_cols, start, yaw0=rng.uniform(-math.pi, math.pi)))))
    return scenes, sensors, reqs


def prepare(case, seed):
    kind = case["kind"]
    st = types.SimpleNamespace(kind=kind, opts=sg.sg_default_opts())
    if kind == "serve":
        scenes, sensors, reqs = _serve_parts(case, seed)
        st.server = Server(n_slots=4)
        st.scenes = {k: sg.Scene(v) for k, v in scenes.items()}
        st.sensors = [sg.Camera(s) if isinstance(s, syn.Camera) else sg.Lidar(s)
                      for s in sensors]
        st.outs, st.poses, st.reqs = [], [], []
        for k, s in reqs:
            if isinstance(s, syn.Camera):
                o = _image(s.height, s.width)
                r = Server.camera_request(st.scenes["camera"], st.sensors[k], s.c2w, o)
            else:
                o = [torch.empty((s.n_beams, s.n_cols), device="cuda") for _ in range(4)]
                st.poses.append(torch.from_numpy(s.col_c2w).cuda())
                r = Server.lidar_request(st.scenes["lidar"], st.sensors[k], st.poses[-1], o)
            st.outs.append(o)
            st.reqs.append(r)
        return st
    src = _scene(case, seed)
    st.scene = sg.Scene(src)
    if kind == "rig":
        st.cams = _rig_cameras(case, seed)
        st.handles = [sg.Camera(c) for c in st.cams]
        st.frames = [_frame(False) for _ in st.cams]
        st.streams = [torch.cuda.Stream() for _ in st.cams]
        st.outs = [_image(c.height, c.width) for c in st.cams]
        st.rows = [torch.from_numpy(c.row_c2w).cuda() if case["rolling"] else None
                   for c in st.cams]
        return st
    if kind in ("lidar", "train_lidar"):
        L = _lidar(case, seed)
        st.sensor = sg.Lidar(L)
        st.poses = torch.from_numpy(L.col_c2w).cuda()
        st.opts = sg.sg_default_opts(beam_divergence=1e-3 * case.get("beam_mrad", 0.0))
        shape = (L.n_beams, L.n_cols)
        ups = dict(range=shape, intensity=shape, drop=shape)
    else:
        cam = _camera(case, seed)
        st.sensor = sg.Camera(cam)
        st.c2w = cam.c2w
        st.rows = torch.from_numpy(cam.row_c2w).cuda() if case.get("rolling") else None
        ups = dict(rgb=(cam.height, cam.width, 3), depth=(cam.height, cam.width))
    if kind == "static":
        st.outs = _image(cam.height, cam.width)
    elif kind in ("camera", "lidar"):
        st.frame = _frame(case["state"])
    else:
        st.frame = sg.Frame()
        st.params = {k: getattr(src, k).requires_grad_() for k in PARAMS}
        st.ups = _upstream(ups, seed)
    return st


# ------------------------------------------------------------------- one pass
def _named(names, outs):
    return dict(zip(names, outs))


CAM_OUT, LID_OUT = ("rgb", "alpha", "depth"), ("range", "intensity", "drop", "alpha")


def run(st):
    if st.kind == "camera":
        if st.rows is None:
            o = sg.render_camera(st.scene, st.sensor, st.c2w, st.opts, st.frame)
        else:
            o = sg.render_camera_rs(st.scene, st.sensor, st.rows, st.opts, st.frame)
        return {k: o[k] for k in CAM_OUT}
    if st.kind == "lidar":
        o = sg.render_lidar(st.scene, st.sensor, st.poses, st.opts, st.frame)
        return {k: o[k] for k in LID_OUT}
    if st.kind == "static":
        sg.sg_render_camera_static(st.scene.handle, st.sensor.handle, st.c2w, st.opts,
                                   *[t.data_ptr() for t in st.outs],
                                   torch.cuda.current_stream().cuda_stream)
        return _named(CAM_OUT, st.outs)
    if st.kind == "rig":
        main = torch.cuda.current_stream()
        for s in st.streams:
            s.wait_stream(main)
        views = sg.sg_camera_views([
            (h.handle, c.c2w, f.handle, o[0].data_ptr(), o[1].data_ptr(), o[2].data_ptr(),
             s.cuda_stream, r.data_ptr() if r is not None else None)
            for h, c, f, o, s, r in zip(st.handles, st.cams, st.frames, st.outs, st.streams,
                                        st.rows)])
        sg.sg_render_cameras(st.scene.handle, views, st.opts, 0)
        for s in st.streams:
            main.wait_stream(s)
        return [_named(CAM_OUT, o) for o in st.outs]
    if st.kind == "serve":
        tickets = [st.server.submit(r) for r in st.reqs]
        for t in tickets:
            st.server.wait(t)
        return [_named(CAM_OUT if len(o) == 3 else LID_OUT, o) for o in st.outs]
    if st.kind == "train_camera":
        outs = _named(CAM_OUT, sga.render_camera(st.params, st.scene, st.sensor, st.c2w,
                                                 st.opts, st.frame))
    else:
        outs = _named(LID_OUT, sga.render_lidar(st.params, st.scene, st.sensor, st.poses,
                                                st.opts, st.frame))
    grads = torch.autograd.grad([outs[k] for k in st.ups], [st.params[k] for k in PARAMS],
                                list(st.ups.values()))
    return dict(outputs={k: v.detach() for k, v in outs.items()}, grads=_named(PARAMS, grads))


# ------------------------------------------------------------------ the floor
def _view_work(n, feats, rays, out_floats, pairs_per_ray):
    """Parameters read once, outputs written once; a projection of seven points (about
    400 operations) a Gaussian and 56 operations an evaluated (ray, Gaussian) pair.  The
    pairs a ray evaluates: the street views' counts at 1M / 2M Gaussians, in proportion
    below that."""
    return (4.0 * (11 + feats) * n + 4.0 * out_floats * rays,
            400.0 * n + 56.0 * pairs_per_ray * rays)


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "serve":
        nc, nl, r = 2 * n // 3, n - 2 * n // 3, case["requests"]
        per = [_view_work(nc, 48, 1920 * 1080, 5, 67.0 * min(1.0, nc / 1e6)),
               _view_work(nc, 48, 1280 * 960, 5, 25.0 * min(1.0, nc / 1e6)),
               _view_work(nl, 3, 64 * 1024, 4, 48.0 * min(1.0, nl / 2e6)),
               _view_work(nl, 3, 128 * 2048, 4, 48.0 * min(1.0, nl / 2e6))]
        b = [per[i % 4] for i in range(r)]
        return dict(bytes=sum(x[0] for x in b), flops=sum(x[1] for x in b))
    if kind in ("lidar", "train_lidar"):
        feats = 3 * (case["degree"] + 1) ** 2 if case["sh"] else 3
        rays = case["beams"] * case["cols"]
        wide = 3.0 if case.get("beam_mrad") else 1.0
        b, f = _view_work(n, feats, rays, 4, 48.0 * wide * min(1.0, n / 2e6))
        ups = 3
    elif kind == "rig":
        feats = 3 * (case["degree"] + 1) ** 2
        k = min(1.0, n / 1e6)
        b, f = (x + y for x, y in zip(_view_work(n, feats, 1920 * 1280, 5, 25.0 * k),
                                      _view_work(n, feats, 1920 * 1080, 5, 67.0 * k)))
    else:
        feats = 3 if case["scene"] == "cube" else 3 * (case["degree"] + 1) ** 2
        rays = case["width"] * case["height"]
        if case["scene"] == "cube":
            per_ray = 20.0 * n / 4096.0
        else:
            per_ray = (25.0 if case["model"] == "fisheye" else 67.0) * min(1.0, n / 1e6)
        b, f = _view_work(n, feats, rays, 5, per_ray)
        ups = 4
    if kind.startswith("train"):   # upstream gradients read, parameter gradients written;
        b += 4.0 * ups * rays + 4.0 * (11 + feats) * n          # about twice the pairs' work
        f *= 3.0
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------- in 64 bits
ALPHA_MIN, ALPHA_MAX = float(np.float32(1.0 / 255.0)), float(np.float32(0.99))
T_MIN, NEAR = float(np.float32(1e-4)), float(np.float32(0.2))
BAND = 12_000_000        # (ray, Gaussian) pairs held at once
F64 = torch.float64


def _d(x):
    return torch.as_tensor(x).to("cuda", F64)


def _mv(A, x):
    """A x for 3x3 matrices A [..., 3, 3] and vectors x [..., 3]."""
    return (A * x[..., None, :]).sum(-1)


def _mtv(A, x):
    """A^T x."""
    return (A * x[..., :, None]).sum(-2)


def _rotation(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x),
                        1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)


def _sh(f, deg, d):
    """sum_k Y_k(d) f_k, real spherical harmonics with the Condon-Shortley phase."""
    x, y, z = d.unbind(1)
    Y = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if deg >= 1:
        a = math.sqrt(3.0 / (4.0 * math.pi))
        Y += [-a * y, a * z, -a * x]
    if deg >= 2:
        a, b, c = (math.sqrt(v / math.pi) for v in (15.0 / 4.0, 5.0 / 16.0, 15.0 / 16.0))
        Y += [a * x * y, -a * y * z, b * (2 * z * z - x * x - y * y), -a * x * z,
              c * (x * x - y * y)]
    if deg >= 3:
        a, b, c, e, h = (math.sqrt(v / math.pi) for v in (35.0 / 32.0, 105.0 / 4.0, 21.0 / 32.0,
                                                          7.0 / 16.0, 105.0 / 16.0))
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (4 * z * z - x * x - y * y),
              e * z * (2 * z * z - 3 * x * x - 3 * y * y), -c * x * (4 * z * z - x * x - y * y),
              h * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return (torch.stack(Y, 1)[:, :, None] * f.reshape(f.shape[0], -1, 3)).sum(1)


class _Params:
    """A scene's parameters in 64 bits (leaves where gradients are asked for) and, in the
    world, its means, rotations and scales."""

    def __init__(self, src, grads):
        self.leaf = {k: getattr(src, k).detach().to(F64).requires_grad_(grads) for k in PARAMS}
        self.kind, self.deg = src.feature_kind, src.sh_degree
        p = self.leaf
        self.mu, self.R, self.s = p["means"], _rotation(p["quats"]), p["log_scales"].exp()
        self.Ra = None
        if src.actor_of is not None:
            P = _d(src.actor_poses).reshape(-1, 3, 4)
            of = torch.as_tensor(src.actor_of).cuda().long()
            eye = torch.eye(3, 4, dtype=F64, device="cuda")[None]
            P = torch.cat([P, eye])[torch.where(of >= 0, of, P.shape[0])]
            self.Ra = P[:, :, :3]
            self.mu = _mv(self.Ra, self.mu) + P[:, :, 3]
            self.R = self.Ra @ self.R

    def features(self, origin):
        """Colour or LiDAR features seen from `origin` ([3] or per Gaussian)."""
        f = self.leaf["features"]
        if self.kind in (syn.FEATURES_RGB, syn.FEATURES_LIDAR):
            return f
        d = self.mu - origin
        d = d / d.norm(dim=1, keepdim=True)
        if self.Ra is not None:
            d = _mtv(self.Ra, d)
        c = _sh(f, self.deg, d)
        return (c + 0.5).clamp(min=0.0) if self.kind == syn.FEATURES_SH else c


def _moments(a):
    """Mean and variance of [n, 7] sigma values: weights (0, 1/6 ..) and (2, 1/6 ..)."""
    m = a[:, 1:].sum(1) / 6.0
    e = (a - m[:, None]) ** 2
    return m, 2.0 * e[:, 0] + e[:, 1:].sum(1) / 6.0


def _sigma_points(mu, D):
    """mu and mu +- sqrt(3) times each column of D."""
    s = math.sqrt(3.0) * D.transpose(1, 2)
    return torch.cat([mu[:, None]] + [x for i in range(3)
                                      for x in ((mu + s[:, i])[:, None], (mu - s[:, i])[:, None])], 1)


def _theta_limit(k):
    r = np.roots([9 * k[3], 7 * k[2], 5 * k[1], 3 * k[0], 1.0])
    r = [x.real for x in r if abs(x.imag) < 1e-12 and 0 < x.real <= (math.pi / 2) ** 2]
    return math.sqrt(min(r)) if r else math.pi / 2


def _pixel(cam, P, x):
    """(u, v, valid) of world points x [..., 3] under poses P [..., 3, 4]."""
    q = _mtv(P[..., :3], x - P[..., 3])
    a, b, z = q.unbind(-1)
    if cam.model == syn.CAMERA_PINHOLE:
        return cam.fx * a / z + cam.cx, cam.fy * b / z + cam.cy, z > NEAR
    k = [float(v) for v in cam.k]
    r = torch.hypot(a, b)
    th = torch.atan2(r, z)
    t2 = th * th
    g = th * (1 + t2 * (k[0] + t2 * (k[1] + t2 * (k[2] + t2 * k[3])))) / r.clamp(min=1e-300)
    return (cam.fx * g * a + cam.cx, cam.fy * g * b + cam.cy,
            (q.norm(dim=-1) > NEAR) & (th <= _theta_limit(k)))


def _pixel_dirs(cam):
    """Camera-frame unit directions [H, W, 3] and which pixels have a ray."""
    x = ((torch.arange(cam.width, device="cuda", dtype=F64) + 0.5 - cam.cx) / cam.fx)[None]
    y = ((torch.arange(cam.height, device="cuda", dtype=F64) + 0.5 - cam.cy) / cam.fy)[:, None]
    x, y = torch.broadcast_tensors(x, y)
    if cam.model == syn.CAMERA_PINHOLE:
        d = torch.stack([x, y, torch.ones_like(x)], 2)
        return d / d.norm(dim=2, keepdim=True), torch.ones_like(x, dtype=torch.bool)
    k, tm = [float(v) for v in cam.k], _theta_limit(cam.k.astype(np.float64))
    rd = torch.hypot(x, y)
    lo, hi = torch.zeros_like(rd), torch.full_like(rd, tm)
    for _ in range(60):       # the model increases on [0, theta_max]
        m = 0.5 * (lo + hi)
        t2 = m * m
        below = m * (1 + t2 * (k[0] + t2 * (k[1] + t2 * (k[2] + t2 * k[3])))) < rd
        lo, hi = torch.where(below, m, lo), torch.where(below, hi, m)
    t = 0.5 * (lo + hi)
    s = torch.sin(t) / rd.clamp(min=1e-300)
    t2 = tm * tm
    limit = tm * (1 + t2 * (k[0] + t2 * (k[1] + t2 * (k[2] + t2 * k[3]))))
    return torch.stack([s * x, s * y, torch.cos(t)], 2), rd <= limit


def _bands(y0, y1, per_row, rows):
    """Row bands [a, b) of at most BAND pairs (a single row may hold more)."""
    diff = torch.zeros(rows + 1, dtype=torch.int64, device="cuda")
    diff.index_add_(0, y0, per_row)
    diff.index_add_(0, y1 + 1, -per_row)
    load = diff.cumsum(0)[:rows].tolist()
    out, a, acc = [], 0, 0
    for r, c in enumerate(load):
        if r > a and acc + c > BAND:
            out.append((a, r))
            a, acc = r, 0
        acc += c
    return out + [(a, rows)]


def _composite(P, seen, box, key, feats, rows, cols, wrap, ray, ups=None):
    """Front-to-back compositing of every ray over the Gaussians whose box holds it.

    seen: indices of the Gaussians, box: their (first column, columns, first row, last
    row), key: float32 distances, feats [n, 3], ray(row, col) -> (origin, direction,
    valid).  Returns sums [rows * cols, 5] (features, Z, W); with `ups`, a function that
    turns a band's sums and ray indices into a scalar loss, its gradients go to the leaves
    of P."""
    dev = "cuda"
    order = torch.sort(key[seen], stable=True).indices
    seen, box = seen[order], [b[order] for b in box]
    x0, nx, y0, y1 = box
    M = (P.R / P.s[:, None, :]).transpose(1, 2)[seen]       # rows of S^-1 R^T, or given
    if getattr(P, "M", None) is not None:
        M = P.M[seen]
    per = [M, P.mu[seen], P.leaf["opacity"][seen], feats[seen]]
    held = [t.detach().requires_grad_(ups is not None) for t in per]
    sums = torch.zeros((rows * cols, 5), dtype=F64, device=dev)

    def pair(g, o, d, t):
        Mg, mu, sig, f = (x[g] for x in t)
        Mv, Md = _mv(Mg, mu - o), _mv(Mg, d)
        dd = (Md * Md).sum(1)
        D2 = (torch.linalg.cross(Mv, Md) ** 2).sum(1) / dd
        return (sig * torch.exp(-0.5 * D2)).clamp(max=ALPHA_MAX), (Mv * Md).sum(1) / dd, f

    for a, b in _bands(y0, y1, nx, rows):
        with torch.no_grad():
            g = torch.nonzero((y0 < b) & (y1 >= a))[:, 0]
            ya, yb = y0[g].clamp(min=a), y1[g].clamp(max=b - 1)
            cnt = nx[g] * (yb - ya + 1)
            total = int(cnt.sum())
            if total == 0:
                continue
            kept = []
            for lo, hi in _chunks(cnt, BAND):
                gg = g[lo:hi].repeat_interleave(cnt[lo:hi])
                off = torch.arange(gg.numel(), device=dev) - (
                    cnt[lo:hi].cumsum(0) - cnt[lo:hi]).repeat_interleave(cnt[lo:hi])
                w = nx[gg]
                r = ya[lo:hi].repeat_interleave(cnt[lo:hi]) + off // w
                c = x0[gg] + off % w
                if wrap:
                    c = c % cols
                o, d, ok = ray(r, c)
                al, tau, _ = pair(gg, o, d, held)
                ok = ok & (tau > 0) & (al >= ALPHA_MIN)
                kept.append((gg[ok], (r * cols + c)[ok], al[ok]))
            gg, idx, al = (torch.cat(z) for z in zip(*kept))
            s = torch.argsort(idx * seen.numel() + gg)
            gg, idx, al = gg[s], idx[s], al[s]
            T = _transmittance(idx, al)
            ok = T * (1 - al) >= T_MIN
            gg, idx = gg[ok], idx[ok]
        if gg.numel() == 0:
            continue
        o, d, _ = ray(idx // cols, idx % cols)
        al, tau, f = pair(gg, o, d, held)
        wgt = al * _transmittance(idx, al)
        q = torch.cat([f, tau[:, None], torch.ones_like(tau)[:, None]], 1) * wgt[:, None]
        first = a * cols
        part = torch.zeros(((b - a) * cols, 5), dtype=F64, device=dev).index_add(0, idx - first, q)
        sums[first:b * cols] = part.detach()
        if ups is not None:
            ups(part, slice(first, b * cols)).backward()
    if ups is not None:
        live = [(t, h.grad) for t, h in zip(per, held) if t.requires_grad and h.grad is not None]
        torch.autograd.backward([t for t, _ in live], [x for _, x in live])
    return sums


def _chunks(cnt, most):
    c, out, lo, base = cnt.cumsum(0).cpu().numpy(), [], 0, 0
    while lo < len(c):
        hi = max(lo + 1, int(np.searchsorted(c, base + most, side="right")))
        out.append((lo, hi))
        lo, base = hi, int(c[hi - 1])
    return out


def _transmittance(idx, al):
    """Product of (1 - alpha) over the earlier entries of the same ray (idx sorted)."""
    c = torch.log1p(-al).cumsum(0)
    c = torch.cat([torch.zeros(1, dtype=F64, device="cuda"), c[:-1]])
    start = torch.ones_like(idx, dtype=torch.bool)
    start[1:] = idx[1:] != idx[:-1]
    at = torch.where(start, torch.arange(idx.numel(), device="cuda"), 0).cummax(0).values
    return torch.exp(c - c[at])


def _exact_camera(src, cam, ups=None):
    P = _Params(src, ups is not None)
    W, H = cam.width, cam.height
    rows = _d(cam.row_c2w if cam.row_c2w is not None else cam.c2w).reshape(-1, 3, 4)
    rolling = cam.row_c2w is not None
    with torch.no_grad():
        pts = _sigma_points(P.mu, P.R * P.s[:, None, :])

        def row_of(x):
            r = torch.full(x.shape[:-1], H // 2 if rolling else 0, dtype=torch.int64,
                           device="cuda")
            for _ in range(2 if rolling else 0):
                _, v, ok = _pixel(cam, rows[r], x)
                r = torch.where(ok, v.nan_to_num(0.0).floor().clamp(0, H - 1).long(), r)
            return r

        u, v, ok = _pixel(cam, rows[row_of(pts)], pts)
        row0 = row_of(P.mu)
        origin = rows[row0][:, :, 3]
        key = (P.mu - origin).norm(dim=1).float()
        sig = P.leaf["opacity"]
        k = torch.sqrt(2 * torch.log((sig / ALPHA_MIN).clamp(min=1.0)))
        (mu_, cu), (mv_, cv) = _moments(u), _moments(v)
        hu, hv = k * cu.sqrt(), k * cv.sqrt()
        ok = ok.all(1) & (sig >= ALPHA_MIN) & torch.isfinite(hu) & torch.isfinite(hv)
        x0 = (mu_ - hu - 0.5).ceil().clamp(0, W)
        x1 = (mu_ + hu - 0.5).floor().clamp(-1, W - 1)
        y0 = (mv_ - hv - 0.5).ceil().clamp(0, H)
        y1 = (mv_ + hv - 0.5).floor().clamp(-1, H - 1)
        ok = ok & (x1 >= x0) & (y1 >= y0)
        seen = torch.nonzero(ok)[:, 0]
        box = [t[seen].long() for t in (x0, x1 - x0 + 1, y0, y1)]
        dirs, valid = _pixel_dirs(cam)

    def ray(r, c):
        pose = rows[r] if rolling else rows
        return pose[:, :, 3], _mv(pose[:, :, :3], dirs[r, c]), valid[r, c]

    loss = None
    if ups is not None:
        g_rgb, g_depth = ups["rgb"].to(F64).reshape(-1, 3), ups["depth"].to(F64).reshape(-1)

        def loss(s, sl):
            hit = s[:, 4] > 0
            depth = torch.where(hit, s[:, 3] / torch.where(hit, s[:, 4], 1.0), 0.0)
            return (s[:, :3] * g_rgb[sl]).sum() + (depth * g_depth[sl]).sum()

    s = _composite(P, seen, box, key, P.features(origin), H, W, False, ray, loss)
    hit = s[:, 4] > 0
    out = dict(rgb=s[:, :3].reshape(H, W, 3), alpha=s[:, 4].reshape(H, W),
               depth=torch.where(hit, s[:, 3] / torch.where(hit, s[:, 4], 1.0), 0.0).reshape(H, W))
    return out, P


def _exact_lidar(src, L, beam=0.0, ups=None):
    P = _Params(src, ups is not None)
    nb, nc, az0 = L.n_beams, L.n_cols, float(L.az0_deg)
    poses = _d(L.col_c2w).reshape(-1, 3, 4)
    elev = _d(L.elevations_deg)
    deg = 180.0 / math.pi

    def see(x):
        c = torch.full(x.shape[:-1], nc // 2, dtype=torch.int64, device="cuda")
        for it in range(3):
            q = _mtv(poses[c][..., :3], x - poses[c][..., 3])
            az = torch.atan2(q[..., 1], q[..., 0]) * deg
            if it < 2:
                c = ((az - az0) * (nc / 360.0)).floor().long() % nc
        r = q.norm(dim=-1)
        return c, az, torch.asin((q[..., 2] / r).clamp(-1, 1)) * deg, r

    with torch.no_grad():
        col0, _, _, r0 = see(P.mu)
        origin = poses[col0][:, :, 3]
        D = P.R * P.s[:, None, :]
        if beam > 0:
            v = P.mu - origin
            C = D @ D.transpose(1, 2) + beam ** 2 * (
                (v * v).sum(1)[:, None, None] * torch.eye(3, dtype=F64, device="cuda")
                - v[:, :, None] * v[:, None, :])
            D = torch.linalg.cholesky(C)
            P.M = torch.linalg.inv(D)
        _, az, el, r = see(_sigma_points(P.mu, D))
        az = torch.where(az - az[:, :1] > 180, az - 360, torch.where(az - az[:, :1] < -180,
                                                                     az + 360, az))
        sig = P.leaf["opacity"]
        k = torch.sqrt(2 * torch.log((sig / ALPHA_MIN).clamp(min=1.0)))
        (ma, ca), (me, ce) = _moments(az), _moments(el)
        ha, he = k * ca.sqrt(), k * ce.sqrt()
        ok = (r > NEAR).all(1) & (sig >= ALPHA_MIN)
        x0 = ((ma - ha - az0) * (nc / 360.0) - 0.5).ceil()
        x1 = ((ma + ha - az0) * (nc / 360.0) - 0.5).floor()
        y0 = torch.searchsorted(elev, (me - he).contiguous())
        y1 = torch.searchsorted(elev, (me + he).contiguous(), right=True) - 1
        ok = ok & (x1 >= x0) & (y1 >= y0)
        seen = torch.nonzero(ok)[:, 0]
        box = [x0[seen].long(), (x1 - x0 + 1).clamp(max=nc)[seen].long(), y0[seen], y1[seen]]

    def ray(b, c):
        a = (az0 + (c.to(F64) + 0.5) * 360.0 / nc) / deg
        e = elev[b] / deg
        u = torch.stack([e.cos() * a.cos(), e.cos() * a.sin(), e.sin()], 1)
        return (poses[c][:, :, 3], _mv(poses[c][:, :, :3], u),
                torch.ones_like(b, dtype=torch.bool))

    def decode(s):
        hit = s[:, 4] > 0
        return (torch.where(hit, s[:, 3] / torch.where(hit, s[:, 4], 1.0), 0.0), s[:, 0],
                torch.sigmoid(s[:, 2] - s[:, 1]), s[:, 4])

    loss = None
    if ups is not None:
        g = [ups[k].to(F64).reshape(-1) for k in LID_OUT[:3]]

        def loss(s, sl):
            return sum((x * y[sl]).sum() for x, y in zip(decode(s), g))

    s = _composite(P, seen, box, r0.float(), P.features(origin), nb, nc, True, ray, loss)
    return {k: v.reshape(nb, nc) for k, v in zip(LID_OUT, decode(s))}, P


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        scenes, _, reqs = _serve_parts(case, seed)
        return [(_exact_camera(scenes["camera"], s) if isinstance(s, syn.Camera)
                 else _exact_lidar(scenes["lidar"], s))[0] for _, s in reqs]
    src = _scene(case, seed)
    if kind == "rig":
        return [_exact_camera(src, c)[0] for c in _rig_cameras(case, seed)]
    if kind == "lidar":
        return _exact_lidar(src, _lidar(case, seed), 1e-3 * case["beam_mrad"])[0]
    if kind == "train_lidar":
        L = _lidar(case, seed)
        shape = (L.n_beams, L.n_cols)
        out, P = _exact_lidar(src, L, 0.0, _upstream(
            dict(range=shape, intensity=shape, drop=shape), seed))
    else:
        cam = _camera(case, seed)
        if kind != "train_camera":
            return _exact_camera(src, cam)[0]
        out, P = _exact_camera(src, cam, _upstream(
            dict(rgb=(cam.height, cam.width, 3), depth=(cam.height, cam.width)), seed))
    return dict(outputs=out, grads={k: P.leaf[k].grad for k in PARAMS})
