"""The work that users of the renderer have it do, as cases to time: renders from one small view to a
batch of 128, a training step, an autograd step, and the side workloads (image randomisation, LiDAR,
mesh transfer, TSDF fusion), each through the public entry points of render.py and dgs.py.

A case is a dict of plain values; `kind` says which part of the library it calls.  Scenes follow the
generators of scenes.py (rooms with posed objects); the sizes are those of its configurations, of
the tests and of bench.py, cut down where building the input would take longer than a second or two.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2507_21981_gb300 import dgs as D
from paper_2507_21981_gb300 import scenes as S
from paper_2507_21981_gb300.render import DeviceScene, GradBuffers, Renderer, render_differentiable

DEVICE = "cuda"
F64 = torch.float64


def listed():
    return [
        # One small plain view: unit tests, thumbnails, the first render of a new asset.  Launches and
        # latency are all of it.
        dict(name="tiny_view", kind="cube", n_bg=8000, n_obj=2000, width=128, height=128, mode="batched"),
        # A control loop with one env and two cameras: the poses of this step go up, the frames come
        # back, a captured graph is replayed.
        dict(name="control_step", kind="room", envs=1, cams=2, n_bg=300_000, n_obj=20_000, objects=4, width=640,
             height=480, dtype="f32", mode="graph", upload=True),
        # The benchmark batch: 64 envs x 2 cameras over a shared million-Gaussian room.
        dict(name="batch_64x2", kind="room", envs=64, cams=2, n_bg=1_000_000, n_obj=20_000, objects=4, width=640,
             height=480, dtype="f32", mode="batched", upload=False),
        # Uneven envs (1-12 assets, 1-3 cameras, three resolutions, odd ones among them), replayed.
        dict(name="ragged_24", kind="ragged", envs=24, n_bg=500_000, assets=16, asset_lo=5_000, asset_hi=100_000,
             w0=317, h0=243, w1=640, h1=480, w2=1271, h2=713, mode="graph"),
        # A larger scene stored in BF16, three cameras per env.
        dict(name="bf16_16x3", kind="room", envs=16, cams=3, n_bg=1_200_000, n_obj=50_000, objects=6, width=640,
             height=480, dtype="bf16", mode="batched", upload=False),
        # Rendering training images: the randomisation (overlay blend, HSV, gamma) fused into the render.
        dict(name="augmented_8x2", kind="augment", envs=8, cams=2, n_bg=200_000, n_obj=20_000, objects=4, width=640,
             height=480, frames=4),
        # Fitting a scene: forward (replayed, lists kept) and backward of one 800x800 view, 500k Gaussians.
        dict(name="train_view_800", kind="train", n_bg=300_000, n_obj=25_000, objects=8, width=800, height=800),
        # The autograd function as an optimiser calls it: four odd-sized views, the backward bins again.
        dict(name="autograd_4_views", kind="autograd", envs=2, cams=2, n_bg=100_000, n_obj=10_000, objects=3,
             width=401, height=301),
        # One spinning LiDAR (32 beams x 1024 azimuths) in a control loop.
        dict(name="lidar_1", kind="lidar", sensors=1, channels=32, azimuths=1024, n_bg=300_000, n_obj=20_000, objects=4),
        # A LiDAR in each of 16 parallel envs.
        dict(name="lidar_16", kind="lidar", sensors=16, channels=32, azimuths=1024, n_bg=500_000, n_obj=20_000,
             objects=4),
        # A scanned mesh (about a million facets, vertex colours) turned into an SH-3 node.
        dict(name="mesh_1m", kind="mesh", nx=709, ny=707, degree=3, colours=True),
        # Fusing 32 depth views into a 256^3 field, as for exporting a node as a mesh.
        dict(name="tsdf_256", kind="tsdf", nx=256, ny=256, nz=256, views=32, width=640, height=480),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cube", "room", "room", "ragged", "augment", "train", "autograd", "lidar", "mesh", "tsdf"])
    if kind == "cube":
        return dict(kind="cube", n_bg=_log_int(rng, 500, 30_000), n_obj=_log_int(rng, 100, 5_000),
                    width=_log_int(rng, 40, 320), height=_log_int(rng, 40, 240), mode=rng.choice(["batched", "graph"]))
    if kind == "room":
        envs = _log_int(rng, 1, 48)
        cams = rng.randint(1, 3 if envs <= 24 else 2)
        w, h = rng.choice([(320, 240), (640, 480), (424, 240), (513, 385), (848, 480)])
        return dict(kind="room", envs=envs, cams=cams, n_bg=_log_int(rng, 50_000, 800_000),
                    n_obj=_log_int(rng, 2_000, 40_000), objects=rng.randint(1, 6), width=w, height=h,
                    dtype=rng.choice(["f32", "f32", "bf16", "f16"]), mode=rng.choice(["batched", "graph"]),
                    upload=rng.random() < 0.5)
    if kind == "ragged":
        (w0, h0), (w1, h1), (w2, h2) = ((rng.randint(a, b), rng.randint(c, d)) for a, b, c, d in
                                        ((100, 330, 80, 250), (400, 650, 300, 490), (700, 1280, 400, 720)))
        return dict(kind="ragged", envs=rng.randint(3, 24), n_bg=_log_int(rng, 50_000, 400_000),
                    assets=rng.randint(4, 16), asset_lo=2_000, asset_hi=60_000, w0=w0, h0=h0, w1=w1, h1=h1, w2=w2,
                    h2=h2, mode=rng.choice(["batched", "graph"]))
    if kind == "augment":
        w, h = rng.choice([(320, 240), (640, 480), (401, 301)])
        return dict(kind="augment", envs=rng.randint(1, 8), cams=2, n_bg=_log_int(rng, 30_000, 200_000),
                    n_obj=_log_int(rng, 2_000, 20_000), objects=rng.randint(1, 4), width=w, height=h,
                    frames=rng.randint(1, 4))
    if kind == "train":
        return dict(kind="train", n_bg=_log_int(rng, 30_000, 300_000), n_obj=_log_int(rng, 2_000, 25_000),
                    objects=rng.randint(1, 8), width=rng.randint(250, 800), height=rng.randint(200, 800))
    if kind == "autograd":
        return dict(kind="autograd", envs=rng.randint(1, 2), cams=rng.randint(1, 2), n_bg=_log_int(rng, 10_000, 100_000),
                    n_obj=_log_int(rng, 500, 10_000), objects=rng.randint(1, 3), width=rng.randint(100, 401),
                    height=rng.randint(80, 301))
    if kind == "lidar":
        return dict(kind="lidar", sensors=rng.randint(1, 8), channels=rng.choice([16, 32, 40, 64]),
                    azimuths=rng.choice([360, 512, 900, 1024]), n_bg=_log_int(rng, 50_000, 400_000),
                    n_obj=_log_int(rng, 2_000, 20_000), objects=rng.randint(1, 4))
    if kind == "mesh":
        return dict(kind="mesh", nx=_log_int(rng, 40, 700), ny=_log_int(rng, 40, 700), degree=rng.randint(0, 3),
                    colours=rng.random() < 0.7)
    return dict(kind="tsdf", nx=rng.randint(50, 250), ny=rng.randint(50, 250), nz=rng.randint(50, 250),
                views=rng.randint(1, 32), width=rng.choice([320, 417, 640]), height=rng.choice([240, 313, 480]))


# ------------------------------------------------------------------------------------------- inputs
def _with_sh3(scene, seed):
    """Degree-3 SH coefficients N(0, 0.2) on every node, the generators' own law, drawn in FP32."""
    rng = np.random.default_rng([seed, 77])
    for nd in scene.nodes:
        nd.sh = rng.standard_normal((nd.n, 16, 3), dtype=np.float32) * np.float32(0.2)
        nd.sh_degree = 3
    return scene


def _ragged_scene(case, seed):
    """Uneven envs in the manner of scenes.config3: which assets (and of which sizes) and cameras an env
    has follows from the case alone, everything else from the seed."""
    E, res = case["envs"], [(case[f"w{i}"], case[f"h{i}"]) for i in range(3)]
    fixed, rng = np.random.default_rng([E, case["assets"], case["n_bg"]]), np.random.default_rng([seed, 78])
    sc = S.config5(seed, n_envs=E, n_bg=case["n_bg"], n_obj=1, n_objects=12, sh_degree=0)   # 12 poses, 3 cameras an env
    sizes = np.exp(fixed.uniform(math.log(case["asset_lo"]), math.log(case["asset_hi"]), case["assets"])).astype(int)
    sc.nodes = sc.nodes[:1] + [S.object_node(rng, int(n), 0) for n in sizes]
    sc.env_node_ids[:, 1:] = -1
    for e in range(E):
        picks = fixed.choice(case["assets"], size=min(int(fixed.integers(1, 13)), case["assets"]), replace=False)
        sc.env_node_ids[e, 1:1 + len(picks)] = np.sort(picks) + 1
        sc.cams_per_env[e] = fixed.integers(1, 4)
        for c in range(3):
            w, h = res[int(fixed.integers(0, 3))]
            sc.cam_res[e, c] = (w, h)
            sc.cam_intr[e, c] = (0.78 * w, 0.78 * w, w / 2.0, h / 2.0)
    return sc


def _scene(case, seed):
    k = case["kind"]
    if k == "cube":
        sc = S.config1(seed, n_bg=case["n_bg"], n_obj=case["n_obj"])
        w, h = case["width"], case["height"]
        f = 110.0 * min(w, h) / 128.0
        sc.cam_res[:] = (w, h)
        sc.cam_intr[:] = (f, f, w / 2.0, h / 2.0)
        return sc
    if k == "ragged":
        return _with_sh3(_ragged_scene(case, seed), seed)
    # every other kind: the room and its objects, one to three cameras per env
    size = dict(n_envs=case.get("envs", case.get("sensors", 1)), n_bg=case["n_bg"], n_obj=case["n_obj"],
                n_objects=case["objects"], width=case.get("width", 640), height=case.get("height", 480), sh_degree=0)
    if case.get("cams", 1) == 3:
        return _with_sh3(S.config5(seed, **size), seed)
    sc = S.config2(seed, **size)
    if k == "train":                   # square pixels, about the field of view of the 800x800 view
        f = 700.0 / 800.0 * max(case["width"], case["height"])
        sc.cam_intr[:, :, 0] = sc.cam_intr[:, :, 1] = f
    sc.cams_per_env[:] = min(case.get("cams", 1), 2)
    return _with_sh3(sc, seed)


def _upstream(ds, seed):
    g = torch.Generator(device=DEVICE).manual_seed(seed * 2 + 1)
    return (torch.randn((ds.n_pixels, 3), generator=g, device=DEVICE),
            torch.randn((ds.n_pixels,), generator=g, device=DEVICE) * 0.3)


def _augmentation(case, seed, n_views):
    clip = S.overlay_frames(seed, n_frames=case["frames"], width=320, height=180)
    prm = S.augment_params(seed, n_views, case["frames"], 320, 180)
    return clip, prm


def _depth_views(case, seed):
    """Depth and coverage of a ball over a floor inside a box-shaped room, from a ring of cameras that
    look at the ball: exact camera-space z of the first surface; a few pixels see nothing (holes)."""
    rng = np.random.default_rng([seed, 55])
    n, w, h = case["views"], case["width"], case["height"]
    f = 0.78 * w
    centre = rng.uniform(-0.1, 0.1, 3)
    radius = rng.uniform(0.3, 0.45)
    ys, xs = torch.meshgrid(torch.arange(h, dtype=F64, device=DEVICE), torch.arange(w, dtype=F64, device=DEVICE),
                            indexing="ij")
    dc = torch.stack([(xs + 0.5 - w / 2) / f, (ys + 0.5 - h / 2) / f, torch.ones_like(xs)], dim=-1)
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    cams, depth, alpha = [], [], []
    for k in range(n):
        az = 2 * math.pi * k / n + rng.uniform(-0.1, 0.1)
        el = rng.uniform(0.2, 0.8)
        eye = centre + rng.uniform(1.4, 1.9) * np.array([math.cos(el) * math.cos(az), math.cos(el) * math.sin(az),
                                                         math.sin(el)])
        P = S.look_at(eye, centre).astype(np.float32)
        R = torch.as_tensor(P[:, :3].astype(np.float64), device=DEVICE)
        e = torch.as_tensor(eye, device=DEVICE)
        d = dc @ R
        oc = e - torch.as_tensor(centre, device=DEVICE)
        a, b = (d * d).sum(-1), 2 * (d @ oc)
        disc = b * b - 4 * a * (oc @ oc - radius * radius)
        z = torch.where(disc > 0, (-b - disc.clamp_min(0).sqrt()) / (2 * a), torch.inf)
        floor = (-0.5 - e[2]) / d[..., 2]
        z = torch.minimum(z, torch.where(floor > 0, floor, torch.inf))
        for ax in (0, 1):                            # walls at +-2.5 m
            z = torch.minimum(z, (torch.sign(d[..., ax]) * 2.5 - e[ax]) / d[..., ax])
        hole = torch.rand((h, w), generator=gen, device=DEVICE) < 0.02
        al = torch.where(hole, 0.2, 0.75 + 0.25 * torch.rand((h, w), generator=gen, device=DEVICE))
        cams.append((f, f, w / 2.0, h / 2.0, w, h, P))
        alpha.append(al.float().reshape(-1))
        depth.append((z * al).float().reshape(-1))
    return cams, torch.cat(depth), torch.cat(alpha)


def _grid(case):
    voxel = 1.2 / max(case["nx"], case["ny"], case["nz"])
    origin = np.array([-0.5 * voxel * case["nx"], -0.5 * voxel * case["ny"], -0.6], np.float32)
    return origin, voxel, 4.0 * voxel


def prepare(case, seed):
    k = case["kind"]
    if k == "mesh":
        v, f, c = S.mesh_heightfield(seed, case["nx"], case["ny"])
        return dict(case=case, r=Renderer(), v=torch.as_tensor(v, device=DEVICE), f=torch.as_tensor(f, device=DEVICE),
                    c=torch.as_tensor(c, device=DEVICE) if case["colours"] else None)
    if k == "tsdf":
        cams, depth, alpha = _depth_views(case, seed)
        shape = (case["nz"], case["ny"], case["nx"])
        return dict(case=case, r=Renderer(), cams=D.cameras(cams), depth=depth, alpha=alpha,
                    F=torch.zeros(shape, device=DEVICE), W=torch.zeros(shape, device=DEVICE))
    ds = DeviceScene(_scene(case, seed), device=DEVICE, dtype=case.get("dtype", "f32"), spatial_order=True)
    st = dict(case=case, ds=ds)
    if k == "lidar":
        st["r"] = Renderer()
        st["r"].lidar_build(ds)
        env, pose = S.lidar_sensors(seed, case["sensors"])
        st["sensors"] = D.lidar_sensors(env, pose)
        st["dirs"] = torch.as_tensor(S.lidar_pattern(case["channels"], case["azimuths"]), device=DEVICE)
    elif k == "train":
        st["r"] = Renderer(mode="graph", keep_lists=1)
        st["grads"] = GradBuffers(ds)
        st["up"] = _upstream(ds, seed)
    elif k == "autograd":
        st["r"] = Renderer()
        for p in ds.param_list():
            p.requires_grad_(True)
        st["poses"] = ds.node_poses.clone().requires_grad_(True)
        st["up"] = _upstream(ds, seed)
    else:
        st["r"] = Renderer(mode=case.get("mode", "batched"))
        if k == "augment":
            clip, prm = _augmentation(case, seed, ds.n_views)
            st["r"].set_augment(prm, torch.as_tensor(clip, device=DEVICE))
        if case.get("upload"):
            st["poses"] = ds.node_poses.cpu().pin_memory()
    return st


def run(state):
    case, r = state["case"], state["r"]
    k = case["kind"]
    if k == "mesh":
        return r.mesh_to_gaussians(state["v"], state["f"], state["c"], sh_degree=case["degree"])
    if k == "tsdf":
        F, W = state["F"].zero_(), state["W"].zero_()
        origin, voxel, trunc = _grid(case)
        rc = D.dgs_tsdf_integrate(r.ctx, F, W, case["nx"], case["ny"], case["nz"], origin, voxel, trunc, 100.0, 0.5,
                                  state["cams"], case["views"], state["depth"], state["alpha"], None,
                                  torch.cuda.current_stream().cuda_stream)
        if rc != D.DGS_OK:
            raise D.DgsError(rc, D.dgs_last_error(r.ctx))
        return F, W
    ds = state["ds"]
    if k == "lidar":
        return r.lidar_trace(ds, state["sensors"], None, state["dirs"])
    if k == "autograd":
        rgb, depth, alpha = render_differentiable(r, ds, state["poses"])
        grads = torch.autograd.grad([rgb, depth], [state["poses"], *ds.param_list()], list(state["up"]))
        return [rgb.detach(), depth.detach(), alpha.detach(), *grads]
    if case.get("upload"):
        ds.set_poses(state["poses"])
    rgb, depth, alpha = r.render(ds)
    if k == "train":
        node_grads, pose_grads = r.backward(ds, rgb, depth, *state["up"], out=state["grads"])
        return [rgb, depth, alpha, pose_grads, *(g[n] for g in node_grads for n in DeviceScene.PARAM_NAMES)]
    return rgb, depth, alpha


# --------------------------------------------------------------------------------------------- work
def work(case):
    """Inputs read once and outputs written once.  Operations: about 300 per Gaussian that a view sees
    (one in eight of those present), and for each pixel the 21 of every Gaussian that covers it before it
    turns opaque (about 40 in these scenes); 50 more for each of those in the adjoint."""
    k = case["kind"]
    if k == "mesh":
        faces, verts = 2 * (case["nx"] - 1) * (case["ny"] - 1), case["nx"] * case["ny"]
        out = 4 * (11 + 3 * (case["degree"] + 1) ** 2)
        return dict(bytes=faces * (12 + out) + verts * (24 if case["colours"] else 12), flops=faces * 120)
    if k == "tsdf":
        vox = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=vox * 16 + case["views"] * case["width"] * case["height"] * 8, flops=vox * case["views"] * 30)
    attr = {"bf16": 16 + 110, "f16": 16 + 110}.get(case.get("dtype"), 236)     # bytes of a stored Gaussian, SH 3
    if k == "cube":
        n, px = case["n_bg"] + case["n_obj"], case["width"] * case["height"]
        return dict(bytes=n * 56 + px * 20, flops=n * 300 + px * 40 * 21)
    if k == "ragged":
        mean = (case["asset_hi"] - case["asset_lo"]) / math.log(case["asset_hi"] / case["asset_lo"])
        n = case["n_bg"] + case["assets"] * mean
        views = 2 * case["envs"]
        px = views * sum(case[f"w{i}"] * case[f"h{i}"] for i in range(3)) / 3
        seen = views * (case["n_bg"] + min(6.5, case["assets"]) * mean) / 8
        return dict(bytes=n * attr + px * 20, flops=seen * 300 + px * 40 * 21)
    n = case["n_bg"] + case["objects"] * case["n_obj"]
    if k == "lidar":
        rays = case["sensors"] * case["channels"] * case["azimuths"]
        return dict(bytes=n * 44 + rays * 8, flops=rays * 40 * 60)
    views = case.get("envs", 1) * case.get("cams", 1)
    px = views * case["width"] * case["height"]
    w = dict(bytes=n * attr + px * 20, flops=views * n / 8 * 300 + px * 40 * 21)
    if k in ("train", "autograd"):     # the upstream gradients read, the attributes read and their gradients written
        w["bytes"] += px * 32 + 2 * n * attr
        w["flops"] += views * n / 8 * 600 + px * 40 * 50
    return w


# ------------------------------------------------------------------- the same results in 64 bits
# Plain torch in FP64.  A view's Gaussians are projected, ordered by (depth, id), listed per 16x16 tile
# by their bounding boxes and composited tile batch by tile batch with cumulative products.
_TILE = 16
_OPT = {k: float(np.float32(v)) for k, v in dict(z_near=0.01, lowpass=0.3, alpha_min=1.0 / 255.0, alpha_max=0.99,
                                                 t_min=1e-4, q_max=9.0, guard=1.3).items()}


def _sh_basis(d):
    x, y, z = d.unbind(-1)
    pi = math.pi
    c1 = math.sqrt(3 / (4 * pi))
    a2, b2, c2 = math.sqrt(15 / (4 * pi)), math.sqrt(5 / (16 * pi)), math.sqrt(15 / (16 * pi))
    a3, b3, c3 = math.sqrt(35 / (32 * pi)), math.sqrt(105 / (4 * pi)), math.sqrt(21 / (32 * pi))
    d3, e3 = math.sqrt(7 / (16 * pi)), math.sqrt(105 / (16 * pi))
    return torch.stack([torch.full_like(x, 0.5 / math.sqrt(pi)), -c1 * y, c1 * z, -c1 * x,
                        a2 * x * y, -a2 * y * z, b2 * (3 * z * z - 1), -a2 * x * z, c2 * (x * x - y * y),
                        -a3 * y * (3 * x * x - y * y), b3 * x * y * z, -c3 * y * (5 * z * z - 1),
                        d3 * z * (5 * z * z - 3), -c3 * x * (5 * z * z - 1), e3 * z * (x * x - y * y),
                        -a3 * x * (x * x - 3 * y * y)], dim=-1)


def _rotation(q):
    w, x, y, z = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], dim=-1).reshape(-1, 3, 3)


def _params64(ds):
    """The stored attributes (rounded as they are stored) in 64 bits, node by node."""
    return [{n: t[n].detach().double() for n in DeviceScene.PARAM_NAMES} for t in ds.tensors]


def _project64(params, env_nodes, poses, cam):
    """Records of the Gaussians in front of the camera and on the image, ordered by depth: (u, v, the
    conic's three entries, opacity, colour, z) and the pixel boxes of their 3-sigma ellipses."""
    fx, fy, cx, cy, W, H, pose = cam
    Wc, tc = pose[:, :3], pose[:, 3]
    recs, boxes = [], []
    for k, slot in sorted((k, j) for j, k in enumerate(env_nodes) if k >= 0):
        g = params[k]
        Rn, tn = poses[slot, :, :3], poses[slot, :, 3]
        M, t0 = Wc @ Rn, Wc @ tn + tc
        mu = g["mean"]
        with torch.no_grad():                          # the few on the image, before anything is built for them
            t = mu @ M.T + t0
            z = t[:, 2]
            smax = torch.exp(g["log_scale"].amax(-1))
            lim = torch.tensor([W, H], device=DEVICE, dtype=F64) * 0.5 * _OPT["guard"] / torch.tensor([fx, fy], device=DEVICE, dtype=F64)
            r = t[:, :2] / z[:, None]
            rc = torch.minimum(torch.maximum(r, -lim), lim)
            ff = torch.tensor([fx, fy], device=DEVICE, dtype=F64)
            c = torch.tensor([cx, cy], device=DEVICE, dtype=F64)
            half = 3.01 * torch.sqrt((ff / z[:, None]) ** 2 * (1 + rc ** 2) * smax[:, None] ** 2 + _OPT["lowpass"]) + 1
            uv = r * ff + c
            wh = torch.tensor([W, H], device=DEVICE, dtype=F64)
            keep = (z > _OPT["z_near"]) & ((uv + half > 0) & (uv - half < wh)).all(-1)
            idx = keep.nonzero().squeeze(1)
        g = {n: p[idx] for n, p in g.items()}
        mu = g["mean"]
        t = mu @ M.T + t0
        z = t[:, 2]
        r = t[:, :2] / z[:, None]
        rc = torch.minimum(torch.maximum(r, -lim), lim)
        J = torch.stack([torch.stack([fx / z, torch.zeros_like(z), -fx * rc[:, 0] / z], -1),
                         torch.stack([torch.zeros_like(z), fy / z, -fy * rc[:, 1] / z], -1)], 1)
        A = (J @ M) @ _rotation(g["quat"]) * torch.exp(g["log_scale"])[:, None, :]
        cxx = (A[:, 0] * A[:, 0]).sum(-1) + _OPT["lowpass"]
        cxy = (A[:, 0] * A[:, 1]).sum(-1)
        cyy = (A[:, 1] * A[:, 1]).sum(-1) + _OPT["lowpass"]
        det = cxx * cyy - cxy * cxy
        uv = r * ff + c
        o = -M.T @ t0
        d = mu - o
        Y = _sh_basis(d / d.norm(dim=-1, keepdim=True))[:, :g["sh"].shape[1]]
        rgb = ((Y[:, :, None] * g["sh"]).sum(1) + 0.5).clamp_min(0)
        recs.append(torch.cat([uv, torch.stack([cyy / det, -cxy / det, cxx / det, torch.sigmoid(g["opacity_logit"])], -1),
                               rgb, z[:, None]], 1))
        boxes.append(torch.sqrt(_OPT["q_max"] * torch.stack([cxx, cyy], -1)).detach())
    rec, half = torch.cat(recs), torch.cat(boxes)
    order = torch.argsort(rec[:, 9].detach(), stable=True)
    return rec[order], half[order]


def _tile_lists(rec, half, W, H):
    """(tiles by descending list length, the start and length of each tile's run, the listed records)."""
    tx, ty = -(-W // _TILE), -(-H // _TILE)
    lim = torch.tensor([W - 1, H - 1], device=DEVICE)
    p0 = torch.ceil(rec[:, :2] - half - 0.5 - 1e-9).long()
    p1 = torch.floor(rec[:, :2] + half - 0.5 + 1e-9).long()
    live = ((p1 >= 0) & (p0 <= lim) & (p0 <= p1)).all(-1)
    p0, p1 = p0.clamp_min(0), torch.minimum(p1, lim)
    t0, t1 = p0 // _TILE, p1 // _TILE
    n = torch.where(live[:, None], t1 - t0 + 1, 0)
    cnt = n[:, 0] * n[:, 1]
    g = torch.repeat_interleave(torch.arange(len(rec), device=DEVICE), cnt)
    k = torch.arange(len(g), device=DEVICE) - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
    tile = (t0[g, 1] + k // n[g, 0].clamp_min(1)) * tx + t0[g, 0] + k % n[g, 0].clamp_min(1)
    tile, perm = torch.sort(tile, stable=True)
    length = torch.bincount(tile, minlength=tx * ty)
    start = torch.cumsum(length, 0) - length
    return torch.argsort(length, descending=True), start, length, g[perm], tx


def _composite64(rec, half, W, H, upstream=None):
    """(rgb, depth, alpha) of one view; with upstream gradients, the records' gradients instead."""
    order, start, length, listed_rec, tx = _tile_lists(rec.detach(), half, W, H)
    out = torch.zeros((H * W, 5), dtype=F64, device=DEVICE)
    pad = torch.zeros((1, 10), dtype=F64, device=DEVICE)
    table = torch.cat([rec.detach(), pad]).requires_grad_(upstream is not None)
    lens = length[order].tolist()
    lane = torch.arange(_TILE * _TILE, device=DEVICE)
    budget = 3_000_000 if upstream is not None else 8_000_000
    at = 0
    while at < len(lens) and lens[at] > 0:
        L = lens[at]
        B = max(1, min(len(lens) - at, budget // (L * 256)))
        tiles = order[at:at + B]
        at += B
        k = torch.arange(L, device=DEVICE)
        idx = torch.where(k < length[tiles, None], start[tiles, None] + k, -1)
        idx = torch.where(idx >= 0, listed_rec[idx.clamp_min(0)], len(rec))
        x = (tiles % tx)[:, None] * _TILE + lane % _TILE
        y = (tiles // tx)[:, None] * _TILE + lane // _TILE
        inside = (x < W) & (y < H)
        with torch.set_grad_enabled(upstream is not None):
            g = table[idx]                                               # [B, L, 10]
            dx = (x + 0.5)[:, None, :] - g[..., 0, None]
            dy = (y + 0.5)[:, None, :] - g[..., 1, None]
            q = g[..., 2, None] * dx * dx + 2 * g[..., 3, None] * dx * dy + g[..., 4, None] * dy * dy
            a = (g[..., 5, None] * torch.exp(-0.5 * q)).clamp_max(_OPT["alpha_max"])
            a = torch.where((q <= _OPT["q_max"]) & (a >= _OPT["alpha_min"]), a, 0.0)
            la = torch.log1p(-a)
            cum = torch.cumsum(la, 1)
            go = torch.cumsum((torch.exp(cum.detach()) < _OPT["t_min"]).int(), 1) == 0
            wgt = torch.where(go, a * torch.exp(cum - la), 0.0)           # [B, L, 256]
            c = torch.einsum("blp,blc->bpc", wgt, g[..., 6:10])
            if upstream is not None:
                p = (y * W + x).clamp_max(W * H - 1)
                up = torch.where(inside[..., None], upstream[p], 0.0)
                (c * up).sum().backward()
                continue
        p = (y * W + x)[inside]
        out[p] = torch.cat([c, wgt.sum(1)[..., None]], -1)[inside]
    if upstream is not None:
        return table.grad[:-1]
    return out[:, :3], out[:, 3], out[:, 4]


def _views(ds):
    sc = ds.scene
    v = 0
    for e in range(sc.n_envs):
        for c in range(int(sc.cams_per_env[e])):
            fx, fy, cx, cy = (float(t) for t in sc.cam_intr[e, c])
            W, H = (int(t) for t in sc.cam_res[e, c])
            pose = torch.as_tensor(sc.cam_pose[e, c].astype(np.float64), device=DEVICE)
            yield v, e, (fx, fy, cx, cy, W, H, pose), slice(int(ds.view_offsets[v]), int(ds.view_offsets[v + 1]))
            v += 1


def _randomise64(rgb, W, prm, clip):
    c = rgb.clamp(0, 1)
    beta = float(prm["overlay_beta"])
    n = len(c)
    i = torch.arange(n, device=DEVICE)
    if beta > 0:
        oh, ow = clip.shape[1:3]
        o = clip[int(prm["overlay_frame"]), (int(prm["overlay_y"]) + i // W) % oh, (int(prm["overlay_x"]) + i % W) % ow]
        c = (1 - beta) * c + beta * o.double() / 255
    r, g, b = c.unbind(-1)
    v, m = c.amax(-1), c.amin(-1)
    d = v - m
    safe = torch.where(d > 0, d, 1.0)
    h = torch.where(v == r, (g - b) / safe, torch.where(v == g, (b - r) / safe + 2, (r - g) / safe + 4))
    h = torch.where(d > 0, torch.remainder(h, 6.0), 0.0)
    s = torch.where(v > 0, d / torch.where(v > 0, v, 1.0), 0.0)
    h = torch.remainder(h + 6 * float(prm["hue_shift"]), 6.0)
    s = (s * float(prm["sat_scale"])).clamp_max(1)
    v = (v * float(prm["val_scale"])).clamp_max(1)
    chan = []
    for k0 in (5, 3, 1):
        k = torch.remainder(k0 + h, 6.0)
        chan.append(v - v * s * torch.minimum(k, 4 - k).clamp(0, 1))
    return torch.stack(chan, -1) ** float(prm["gamma"])


def _exact_render(case, seed):
    ds = DeviceScene(_scene(case, seed), device=DEVICE, dtype=case.get("dtype", "f32"), spatial_order=True)
    if ds.n_views > 64:
        return None                                      # over 20 seconds
    grads = case["kind"] in ("train", "autograd")
    params = _params64(ds)
    poses = ds.node_poses.double().reshape(ds.n_envs, ds.max_nodes, 3, 4)
    if grads:
        poses.requires_grad_(True)
        for g in params:
            for p in g.values():
                p.requires_grad_(True)
        up = torch.cat([t.reshape(ds.n_pixels, -1).double() for t in _upstream(ds, seed)], 1)
    if case["kind"] == "augment":
        clip, prm = _augmentation(case, seed, ds.n_views)
        clip = torch.as_tensor(clip, device=DEVICE)
    out = [torch.zeros((ds.n_pixels, 3), dtype=F64, device=DEVICE), torch.zeros(ds.n_pixels, dtype=F64, device=DEVICE),
           torch.zeros(ds.n_pixels, dtype=F64, device=DEVICE)]
    for v, e, cam, px in _views(ds):
        with torch.set_grad_enabled(grads):
            rec, half = _project64(params, [int(k) for k in ds.env_node_ids[e]], poses[e], cam)
        with torch.no_grad():
            rgb, depth, alpha = _composite64(rec, half, cam[4], cam[5])
        if case["kind"] == "augment":
            rgb = _randomise64(rgb, cam[4], prm[v], clip)
        out[0][px], out[1][px], out[2][px] = rgb, depth, alpha
        if grads:
            rec.backward(_composite64(rec, half, cam[4], cam[5], up[px]))
    if not grads:
        return tuple(out)
    g_pose = poses.grad
    flat = [p.grad if p.grad is not None else torch.zeros_like(p) for g in params for p in g.values()]
    if case["kind"] == "autograd":
        g_pose = g_pose.reshape(ds.node_poses.shape)
    return [*out, g_pose, *flat]


def _exact_lidar(case, seed):
    ds = DeviceScene(_scene(case, seed), device=DEVICE, spatial_order=True)
    env, pose = S.lidar_sensors(seed, case["sensors"])
    dirs = torch.as_tensor(S.lidar_pattern(case["channels"], case["azimuths"]), device=DEVICE).double()
    dirs = dirs / dirs.norm(dim=-1, keepdim=True)
    params = _params64(ds)
    nodes = []
    for g in params:
        s = torch.exp(g["log_scale"])
        nodes.append((g["mean"], _rotation(g["quat"]).transpose(1, 2) / s[:, :, None], torch.sigmoid(g["opacity_logit"]),
                      (3.001 * s.amax(-1)) ** 2))
    J = len(dirs)
    D_out = torch.zeros((case["sensors"], J), dtype=F64, device=DEVICE)
    A_out = torch.zeros_like(D_out)
    r_min, r_max = float(np.float32(0.05)), 30.0
    gbase = np.concatenate([[0], np.cumsum([len(n[0]) for n in nodes])])
    for i in range(case["sensors"]):
        Ws = torch.as_tensor(pose[i].astype(np.float64), device=DEVICE)
        ray, ts, al, gid = [], [], [], []
        for j, k in enumerate(int(k) for k in ds.env_node_ids[int(env[i])]):
            if k < 0:
                continue
            mean, M, op, rad2 = nodes[k]
            Wn = ds.node_poses[int(env[i]), j].double().reshape(3, 4)
            R = Wn[:, :3].T @ Ws[:, :3]
            o = Wn[:, :3].T @ (Ws[:, 3] - Wn[:, 3])
            d = dirs @ R.T
            vec = mean - o
            vv = (vec * vec).sum(-1)
            step = max(1, 60_000_000 // J)
            for a in range(0, len(mean), step):
                v = vec[a:a + step]
                b = v @ d.T                                               # [Gaussians, rays]
                near = (vv[a:a + step, None] - b * b <= rad2[a:a + step, None]) & (b > -1)
                gi, ri = near.nonzero(as_tuple=True)
                gi = gi + a
                op_ = -torch.einsum("nab,nb->na", M[gi], vec[gi])
                dp = torch.einsum("nab,nb->na", M[gi], d[ri])
                dd = (dp * dp).sum(-1)
                t = -(op_ * dp).sum(-1) / dd
                q = (torch.linalg.cross(op_, dp) ** 2).sum(-1) / dd
                alpha = (op[gi] * torch.exp(-0.5 * q)).clamp_max(_OPT["alpha_max"])
                ok = (q <= _OPT["q_max"]) & (t >= r_min) & (t <= r_max) & (alpha >= _OPT["alpha_min"])
                ray.append(ri[ok]); ts.append(t[ok]); al.append(alpha[ok]); gid.append(gi[ok] + int(gbase[k]))
        ray, ts, al, gid = (torch.cat(x) for x in (ray, ts, al, gid))
        p = torch.argsort(gid)                                            # by ray, then distance, then id
        p = p[torch.argsort(ts[p], stable=True)]
        p = p[torch.argsort(ray[p], stable=True)]
        ray, ts, al = ray[p], ts[p], al[p]
        cnt = torch.bincount(ray, minlength=J)
        start = torch.cumsum(cnt, 0) - cnt
        la = torch.log1p(-al)
        cum = torch.cumsum(la, 0)
        before = (cum - la)[start.clamp_max(max(len(cum) - 1, 0))] if len(cum) else torch.zeros(J, dtype=F64, device=DEVICE)
        rel = cum - before[ray]
        stop = (torch.exp(rel) < _OPT["t_min"]).long()
        cs = torch.cumsum(stop, 0)
        ok = cs - (cs - stop)[start.clamp_max(max(len(cum) - 1, 0))][ray] == 0
        w = torch.where(ok, al * torch.exp(rel - la), 0.0)
        D_out[i].index_add_(0, ray, w * ts)
        A_out[i].index_add_(0, ray, w)
    return D_out, A_out


def _exact_mesh(case, seed):
    v, f, col = S.mesh_heightfield(seed, case["nx"], case["ny"])
    v, col = (torch.as_tensor(x, device=DEVICE).double() for x in (v, col))
    f = torch.as_tensor(f, device=DEVICE).long()
    p = v[f]
    bc = p.mean(1)
    s = (p - bc[:, None]).norm(dim=-1).mean(1)
    t1 = torch.nn.functional.normalize(p[:, 1] - p[:, 0], dim=-1)
    n = torch.nn.functional.normalize(torch.linalg.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]), dim=-1)
    R = torch.stack([t1, torch.linalg.cross(n, t1), n], -1)
    tr = R.diagonal(dim1=1, dim2=2)
    trace = tr.sum(-1)
    # the quaternion's outer product 4 q q^T from the rotation: take its row with the largest diagonal
    x, y, z = tr.unbind(-1)
    d21, d02, d10 = R[:, 2, 1] - R[:, 1, 2], R[:, 0, 2] - R[:, 2, 0], R[:, 1, 0] - R[:, 0, 1]
    s10, s20, s21 = R[:, 1, 0] + R[:, 0, 1], R[:, 2, 0] + R[:, 0, 2], R[:, 2, 1] + R[:, 1, 2]
    K = torch.stack([torch.stack([1 + trace, d21, d02, d10], -1), torch.stack([d21, 1 + x - y - z, s10, s20], -1),
                     torch.stack([d02, s10, 1 - x + y - z, s21], -1), torch.stack([d10, s20, s21, 1 - x - y + z], -1)], 1)
    row = K.diagonal(dim1=1, dim2=2).argmax(-1)
    q = torch.nn.functional.normalize(K[torch.arange(len(K), device=DEVICE), row], dim=-1)
    q = torch.where(q[:, :1] < 0, -q, q)
    flat = float(np.float32(0.01))
    sh = torch.zeros((len(f), (case["degree"] + 1) ** 2, 3), dtype=F64, device=DEVICE)
    if case["colours"]:
        sh[:, 0] = (col[f].mean(1) - 0.5) * 2 * math.sqrt(math.pi)
    return dict(mean=bc, log_scale=torch.stack([s.log(), s.log(), (flat * s).log()], -1), quat=q,
                opacity_logit=torch.full((len(f),), 2.0, dtype=F64, device=DEVICE), sh=sh)


def _exact_tsdf(case, seed):
    cams, depth, alpha = _depth_views(case, seed)
    origin, voxel, trunc = _grid(case)
    voxel, trunc = float(np.float32(voxel)), float(np.float32(trunc))
    ax = [float(origin[a]) + (torch.arange(n, device=DEVICE, dtype=F64) + 0.5) * voxel
          for a, n in enumerate((case["nx"], case["ny"], case["nz"]))]
    z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    F, Wt = torch.zeros_like(x), torch.zeros_like(x)
    n = case["width"] * case["height"]
    for k, (fx, fy, cx, cy, w, h, P) in enumerate(cams):
        P = P.astype(np.float64)
        fx, fy = float(np.float32(fx)), float(np.float32(fy))
        xc, yc, zc = (P[a, 0] * x + P[a, 1] * y + P[a, 2] * z + P[a, 3] for a in range(3))
        u, v = fx * xc / zc + cx, fy * yc / zc + cy
        ok = (zc > 0) & (u >= 0) & (v >= 0) & (u < w) & (v < h)
        p = torch.where(ok, v.floor() * w + u.floor(), 0.0).long()
        d, a = depth[k * n:(k + 1) * n].double()[p], alpha[k * n:(k + 1) * n].double()[p]
        sdf = d / a - zc
        ok &= (a >= 0.5) & (sdf >= -trunc)
        F = torch.where(ok, (Wt * F + (sdf / trunc).clamp_max(1)) / (Wt + 1), F)
        Wt = torch.where(ok, (Wt + 1).clamp_max(100.0), Wt)
    return F, Wt


def exact(case, seed):
    k = case["kind"]
    if k == "lidar":
        if case["sensors"] * case["channels"] * case["azimuths"] * (case["n_bg"] + case["objects"] * case["n_obj"]) > 4e11:
            return None                                  # over 20 seconds
        return _exact_lidar(case, seed)
    if k == "mesh":
        return _exact_mesh(case, seed)
    if k == "tsdf":
        return _exact_tsdf(case, seed)
    return _exact_render(case, seed)
