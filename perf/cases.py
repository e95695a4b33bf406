"""What is measured of this framework: the calls a frame-to-map RGB-D system
makes into it, at the sizes of the repository's own benchmark and tests.

Per frame: the tracking loop (gs2d_track_step), optionally started by the
learned proposal, and the keyframe test.  Per keyframe: the map expansion,
the map-state passes and mapping steps over a window or an uneven batch of
views.  Offline: training of the proposal network.  Observed frames are ray
casts of the synthetic room whose surfels form the map, so no input depends
on the renderer.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2506_00970_gb300 import gs2d, proposal, scenes

DEV = "cuda"
N_KF = 64                       # keyframes of the map-state case
BLENDED = 19                    # blended (pixel, surfel) pairs per pixel of a room view
CONV = (8, 32, 64, 128, 256, 256, 256)


def listed():
    return [
        # the smallest optimisation step: a thumbnail view of a few thousand surfels
        dict(name="slab_160x120", kind="single", n=4096, w=160, h=120, f=150.0),
        # coarse-to-fine tracking: a room map seen by the proposal network's small camera
        dict(name="track_160x120", kind="track", n=200_000, w=160, h=120, f=150.0, iters=10),
        # tracking of a VGA sensor frame, the per-frame work of the system
        dict(name="track_640x480", kind="track", n=200_000, w=640, h=480, f=525.0, iters=10),
        # keyframe test of a cropped (undistorted) VGA frame: ragged edges in both directions
        dict(name="keyframe_633x471", kind="keyframe", n=200_000, w=633, h=471, f=525.0),
        # a mapping step over a window of eight keyframes
        dict(name="window_8x1200x680", kind="window", n=1_000_000, views=8, w=1200, h=680, f=600.0),
        # a mapping step over 32 keyframes of mixed resolution, each with its own active map
        dict(name="uneven_32", kind="uneven", n=2_000_000, views=32, lo=50_000, hi=1_000_000),
        # the whole learned proposal of one frame: two renders-and-network passes
        dict(name="proposal_160x120", kind="proposal", n=200_000, passes=2),
        # one training step of the proposal network
        dict(name="net_train_256", kind="train", batch=256),
        # proposals for a queue of frames, an odd batch
        dict(name="net_forward_77", kind="forward", batch=77),
        # the map-state passes after a keyframe of a large map
        dict(name="map_2m", kind="map", n=2_000_000),
        # new surfels of a keyframe against the voxel table of the active map
        dict(name="expand_1200x680", kind="expand", n=1_000_000, w=1200, h=680, f=600.0, ratio=0.04),
        # the full mapping loss with its SSIM term of one keyframe
        dict(name="ssim_loss_1200x680", kind="ssim", w=1200, h=680, f=600.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single", "track", "track", "keyframe", "window", "uneven", "proposal",
                       "train", "forward", "map", "expand", "ssim"])
    c = dict(kind=kind)
    if kind in ("single", "track", "keyframe", "expand", "ssim", "window"):
        lo, hi = {"single": (96, 320), "track": (120, 660), "keyframe": (300, 660),
                  "expand": (300, 1200), "ssim": (160, 1280), "window": (320, 1200)}[kind]
        c["w"] = _log(rng, lo, hi)
        c["h"] = max(61, min(720, int(c["w"] * rng.uniform(0.56, 0.8))))
        c["f"] = round(c["w"] * rng.uniform(0.5, 0.95), 2)
    if kind == "single":
        c["n"] = _log(rng, 1_000, 40_000)
    elif kind == "track":
        c["n"], c["iters"] = _log(rng, 40_000, 300_000), rng.randint(3, 10)
    elif kind == "keyframe":
        c["n"] = _log(rng, 50_000, 400_000)
    elif kind == "window":
        c["n"], c["views"] = _log(rng, 150_000, 1_000_000), rng.randint(2, 8)
    elif kind == "uneven":
        c["n"], c["views"] = _log(rng, 400_000, 2_000_000), rng.randint(3, 32)
        c["lo"], c["hi"] = 30_000, max(100_000, c["n"] // 2)
    elif kind == "proposal":
        c["n"], c["passes"] = _log(rng, 50_000, 300_000), rng.randint(1, 2)
    elif kind == "train":
        c["batch"] = _log(rng, 16, 256)
    elif kind == "forward":
        c["batch"] = _log(rng, 1, 256)
    elif kind == "map":
        c["n"] = _log(rng, 30_000, 2_000_000)
    elif kind == "expand":
        c["n"], c["ratio"] = _log(rng, 50_000, 1_000_000), round(rng.uniform(0.01, 0.06), 4)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 7919 + 17)
    return g


def _t(a, dtype=torch.float32):
    return torch.as_tensor(np.asarray(a), dtype=dtype, device=DEV)


class _Room:
    """The surfaces of a synthetic room: surfels sampled on them, and ray
    casts of them."""

    def __init__(self, seed):
        self.p = scenes._room_patches(np.random.default_rng(seed))

    def surfels(self, n, g):
        p = self.p
        z = np.zeros(3)
        areas = _t([q.area for q in p], torch.float64)
        k = torch.multinomial(areas, n, replacement=True, generator=g)
        rect = _t([q.kind == "rect" for q in p], torch.bool)[k][:, None]
        col = lambda f: _t([f(q) for q in p])[k]
        a, b = torch.rand(n, 1, generator=g, device=DEV), torch.rand(n, 1, generator=g, device=DEV)
        d = F.normalize(torch.randn(n, 3, generator=g, device=DEV), dim=1)
        r = lambda q, v: v if q.kind == "rect" else z
        s = lambda q, v: v if q.kind != "rect" else z
        mu = torch.where(rect, col(lambda q: r(q, q.origin)) + a * col(lambda q: r(q, q.e1))
                         + b * col(lambda q: r(q, q.e2)),
                         col(lambda q: s(q, q.centre)) + col(lambda q: [q.radius]) * d)
        tn = torch.where(rect, col(lambda q: r(q, q.normal)), -d)
        # a random frame with t_n as its third axis, as a quaternion: the shortest rotation of
        # the z axis onto t_n after a random turn about z
        up = tn[:, 2:] > -0.9
        h = torch.where(up, torch.cat([1 + tn[:, 2:], -tn[:, 1:2], tn[:, :1], torch.zeros_like(a)], 1),
                        torch.cat([-tn[:, 1:2], 1 - tn[:, 2:], torch.zeros_like(a), tn[:, :1]], 1))
        h = F.normalize(h, dim=1)
        phi = math.pi * torch.rand(n, 1, generator=g, device=DEV)
        c, sn = torch.cos(phi), torch.sin(phi)
        w, x, y, v = h.split(1, 1)
        quat = torch.cat([w * c - v * sn, x * c + y * sn, y * c - x * sn, v * c + w * sn], 1)
        scale = 0.01 + 0.02 * torch.rand(n, 2, generator=g, device=DEV)
        rgb = (col(lambda q: q.albedo) + 0.03 * torch.randn(n, 3, generator=g, device=DEV)).clamp(0, 1)
        return [mu, quat, scale, torch.full((n,), 0.9, device=DEV), rgb]

    def cast(self, cam, pose, g, noise=0.001, holes=0.02):
        """(rgb, depth, normal) of the first surface along each pixel ray:
        sensor noise on colour and depth, depth 0 at a few holes; the normal
        in the camera frame points into the material."""
        f8 = dict(dtype=torch.float64, device=DEV)
        R, t = _t(pose.R, torch.float64), _t(pose.t, torch.float64)
        x = (torch.arange(cam.width, **f8) + 0.5 - cam.cx) / cam.fx
        y = (torch.arange(cam.height, **f8) + 0.5 - cam.cy) / cam.fy
        ray = torch.stack(torch.meshgrid(x, y, indexing="xy") + (torch.ones(cam.height, cam.width, **f8),), -1)
        d, eye = ray @ R, -(R.T @ t)
        best = torch.full((cam.height, cam.width), 1e9, **f8)
        rgb, nrm = torch.zeros(cam.height, cam.width, 3, **f8), torch.zeros(cam.height, cam.width, 3, **f8)
        for q in self.p:
            if q.kind == "rect":
                o, e1, e2, n = (_t(v, torch.float64) for v in (q.origin, q.e1, q.e2, q.normal))
                dist = ((o - eye) @ n) / (d @ n)
                X = eye + dist[..., None] * d - o
                a, b = X @ e1 / (e1 @ e1), X @ e2 / (e2 @ e2)
                ok = (dist > 0.05) & (a >= 0) & (a <= 1) & (b >= 0) & (b <= 1)
                n = n.expand_as(d)
            else:
                o = _t(q.centre, torch.float64) - eye
                A, B = (d * d).sum(-1), d @ o
                disc = B * B - A * (o @ o - q.radius ** 2)
                dist = (B - disc.clamp_min(0).sqrt()) / A
                ok = (disc > 0) & (dist > 0.05)
                n = (o - dist[..., None] * d) / q.radius
            ok = ok & (dist < best)
            best = torch.where(ok, dist, best)
            rgb = torch.where(ok[..., None], _t(q.albedo, torch.float64), rgb)
            nrm = torch.where(ok[..., None], n, nrm)
        depth = best + noise * torch.randn(best.shape, generator=g, **f8)
        depth = torch.where(torch.rand(best.shape, generator=g, **f8) < holes, 0.0, depth)
        rgb = (rgb + 0.02 * torch.randn(rgb.shape, generator=g, **f8)).clamp(0, 1)
        return rgb.float(), depth.float(), (nrm @ R.T).float()


def _cam(c):
    return scenes.Camera(c["f"], c["f"], c["w"] / 2, c["h"] / 2, c["w"], c["h"])


def _views(case, seed):
    """Cameras, poses and active-subset sizes of a batch case."""
    v = case["views"]
    if case["kind"] == "window":
        return [_cam(case)] * v, scenes.room_trajectory(seed, v), [None] * v
    rng = np.random.default_rng(seed)
    cams = scenes.uneven_cameras(seed, v)
    poses = [scenes.room_pose(1000 * seed + k) for k in range(v)]
    size = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), v)).astype(int)
    return cams, poses, [min(int(s), case["n"]) for s in size]


def _inputs(case, seed):
    """Every input tensor of a case, the same for every build."""
    g, k = _gen(seed), case["kind"]
    i = {}
    if k == "single":
        s = scenes.slab_scene(seed, case["n"])
        i["surf"] = [_t(a) for a in (s.mu, s.quat, s.scale, s.opacity, s.rgb)]
        i["cam"], i["pose"] = _cam(case), scenes.identity_pose()
        i["obs"] = [_t(a) for a in scenes.rgbd_frame(seed, i["cam"])]
    elif k in ("track", "keyframe", "proposal"):
        room = _Room(seed)
        i["surf"] = room.surfels(case["n"], g)
        i["cam"] = proposal.CAM if k == "proposal" else _cam(case)
        gt = scenes.room_pose(100 + seed)
        trans, rot = (0.05, 2.0) if k == "keyframe" else (0.02, 1.0)
        i["pose"] = scenes.perturb_pose(gt, trans, rot, seed=5000 + seed)
        i["kf_pose"] = gt
        if k == "keyframe":
            # the last keyframe's contributions: a random weight for what lies in its view
            X = i["surf"][0] @ _t(gt.R).T + _t(gt.t)
            x, y = X[:, 0] / X[:, 2], X[:, 1] / X[:, 2]
            seen = (X[:, 2] > 0.05) & (x.abs() < case["w"] / 2 / case["f"]) & (y.abs() < case["h"] / 2 / case["f"])
            i["c_kf"] = seen * 3 * torch.rand(case["n"], generator=g, device=DEV)
        else:
            i["obs"] = room.cast(i["cam"], gt, g)[:2]
        if k == "proposal":
            i["params"] = _net_params(g)
    elif k in ("window", "uneven"):
        room = _Room(seed)
        s = room.surfels(case["n"], g)
        i["cams"], i["poses"], sizes = _views(case, seed)
        i["obs"] = [room.cast(c, p, g)[:2] for c, p in zip(i["cams"], i["poses"])]
        i["actives"] = []
        for p, m in zip(i["poses"], sizes):
            if m is None:
                i["actives"].append(None)
                continue
            ahead = _t(-p.R.T @ p.t + 1.5 * p.R[2])
            ids = torch.topk(((s[0] - ahead) ** 2).sum(1), m, largest=False).indices
            i["actives"].append(ids.sort().values.to(torch.int32))
        # the map under optimisation is a little off the surfaces
        s[0] = s[0] + 0.003 * torch.randn(s[0].shape, generator=g, device=DEV)
        s[4] = s[4] + 0.05 * torch.randn(s[4].shape, generator=g, device=DEV)
        i["surf"] = s
    elif k in ("train", "forward"):
        B = case["batch"]
        # rendered and observed RGB-D: smooth surfaces with sensor noise
        low = torch.rand(B, 8, 12, 16, generator=g, device=DEV)
        x = F.interpolate(low, (120, 160), mode="bilinear").permute(0, 2, 3, 1)
        x = x + 0.03 * torch.randn(x.shape, generator=g, device=DEV)
        span = _t([1, 1, 1, 3, 1, 1, 1, 3])
        i["x"] = ((x - 0.5) * span + _t([0.5, 0.5, 0.5, 0, 0.5, 0.5, 0.5, 0])).to(torch.bfloat16).contiguous()
        i["params"] = _net_params(g)
        if k == "train":
            P = i["params"].numel()
            i["target"] = 0.7 * torch.randn(B, 6, generator=g, device=DEV)
            i["m"] = 1e-3 * torch.randn(P, generator=g, device=DEV)
            i["v"] = 1e-6 * (0.1 + torch.rand(P, generator=g, device=DEV))
    elif k == "map":
        n = case["n"]
        s = _Room(seed).surfels(n, g)
        i["surf"] = s
        levels = _t([0.0, 0.0, 0.0, 0.3, 0.7, 2.0])
        i["contrib"] = levels[torch.randint(0, 6, (n,), generator=g, device=DEV)]
        i["delta"] = (torch.rand(n, generator=g, device=DEV) < 0.8).to(torch.uint8)
        i["t_c"] = torch.randint(0, N_KF, (n,), generator=g, device=DEV, dtype=torch.int32)
        i["t_l"] = torch.randint(N_KF - 30, N_KF, (n,), generator=g, device=DEV, dtype=torch.int32)
        i["d_c"] = 0.5 + 3 * torch.rand(n, generator=g, device=DEV)
        i["pose"] = scenes.room_pose(seed + 5)
        old = scenes.room_trajectory(seed, N_KF)
        new = [scenes.perturb_pose(p, 0.03, 0.5, seed=seed + j) for j, p in enumerate(old)]
        i["old"], i["new"] = (torch.stack([gs2d.pose_tensor(p, DEV) for p in q]) for q in (old, new))
    elif k == "expand":
        room = _Room(seed)
        i["cam"], i["pose"] = _cam(case), scenes.room_pose(seed + 3)
        i["rgb"], i["depth"], _ = room.cast(i["cam"], i["pose"], g)
        # the active map covers the far half of the room's length, a few mm off the surfaces
        act = room.surfels(2 * case["n"], g)[0]
        act = act + 0.003 * torch.randn(act.shape, generator=g, device=DEV)
        i["act"] = act[act[:, 0] > scenes.ROOM[0] / 2][:case["n"]].contiguous()
        i["u_keep"], i["u_angle"] = (torch.rand(case["h"], case["w"], generator=g, device=DEV) for _ in range(2))
    elif k == "ssim":
        room, i["cam"] = _Room(seed), _cam(case)
        rgb, depth, nrm = room.cast(i["cam"], scenes.room_pose(seed), g)
        op = (0.97 + 0.03 * torch.rand(depth.shape, generator=g, device=DEV))
        op = torch.where(torch.rand(depth.shape, generator=g, device=DEV) < 0.01, 0.4, op)
        noise = lambda a, s: a + s * torch.randn(a.shape, generator=g, device=DEV)
        i["obs"] = [rgb, depth]
        i["ren"] = [noise(rgb, 0.05).clamp(0, 1) * op[..., None], noise(depth.clamp_min(0.3), 0.004) * op,
                    F.normalize(noise(nrm, 0.05), dim=-1) * op[..., None], op]
        i["ren"] = [a.contiguous() for a in i["ren"]]
    return i


def _net_params(g):
    parts = []
    for ci, co in list(zip(CONV[:-1], CONV[1:])) + [(1536 / 9, 256), (256 / 9, 6)]:
        fan = int(round(9 * ci))
        parts += [math.sqrt(2 / fan) * torch.randn(co * fan, generator=g, device=DEV),
                  0.05 * torch.randn(co, generator=g, device=DEV)]
    return torch.cat(parts)


# ---------------------------------------------------------------------------
# what a program holds before the call, and the call
# ---------------------------------------------------------------------------
def _bytes(n):
    return torch.empty(max(int(n), 1), dtype=torch.uint8, device=DEV)


def prepare(case, seed):
    i, k = _inputs(case, seed), case["kind"]
    st = dict(i, case=case)
    if "surf" in i:
        st["ds"] = gs2d.DeviceSurfels.from_tensors(*i["surf"])
    if "cam" in i:
        st["ccam"] = gs2d.camera(i["cam"])
    z = lambda *s, dt=torch.float32: torch.zeros(*s, dtype=dt, device=DEV)
    if "pose" in i:
        st["pose_t"] = gs2d.pose_tensor(i["pose"], DEV)
    if k == "single":
        st["r"] = gs2d.Rasterizer(i["cam"], case["n"])
        h, w = case["h"], case["w"]
        st["g"] = [z(h, w, 3), z(h, w), z(h, w, 3), z(h, w)]
        st["loss"], st["lws"] = z(1), _bytes(1 << 16)
    elif k == "track":
        st["cfg"], st["prm"] = gs2d.default_config(), gs2d.default_track_params(stop_tol=0.0)
        st["cap"] = 8 * case["n"]
        st["ws"] = _bytes(gs2d.gs2d_track_workspace(case["n"], st["cap"], st["ccam"], st["cfg"]))
        it = case["iters"]
        st["cur"], st["loss"], st["poses"], st["grads"] = z(12), z(it), z(it, 12), z(it, 6)
    elif k == "keyframe":
        st["r"] = gs2d.Rasterizer(i["cam"], case["n"], capacity=8 * case["n"])
        st["kf_t"] = gs2d.pose_tensor(i["kf_pose"], DEV)
        st["contrib"], st["score"] = z(case["n"]), z(1)
        st["counts"], st["is_kf"] = z(2, dt=torch.int32), z(1, dt=torch.int32)
    elif k in ("window", "uneven"):
        br = gs2d.BatchRasterizer(i["cams"], case["n"],
                                  actives=[None if a is None else a.cpu().numpy() for a in i["actives"]])
        br.set_poses(i["poses"])
        br.fit(st["ds"])
        st["br"], st["loss"] = br, z(len(i["cams"]))
        st["lv"] = gs2d.loss_views([(b["ccam"], b["rgb"], b["depth"], b["normal"], b["opacity"], o[0], o[1],
                                     b["d_rgb"], b["d_depth"], b["d_normal"], b["d_opacity"])
                                    for b, o in zip(br.keep, i["obs"])])
        st["lws"] = _bytes(gs2d.gs2d_mapping_loss_batch_workspace(st["lv"]))
    elif k == "proposal":
        pr = proposal.Proposer(st["ds"], i["params"], 8 * case["n"], passes=case["passes"])
        pr.pose.copy_(st["pose_t"][None])
        pr.obs_rgb.copy_(i["obs"][0])
        pr.obs_d.copy_(i["obs"][1])
        st["pr"], st["graph"] = pr, proposal.capture(pr.run)
    elif k in ("train", "forward"):
        B = case["batch"]
        st["ws"], st["y"] = _bytes(gs2d.gs2d_net_workspace(B)), z(B, 6)
        if k == "train":
            st["grad"], st["loss"], st["step"] = z(i["params"].numel()), z(1), 100
        else:
            gs2d.gs2d_net_prepare(i["params"], B, st["ws"])
    elif k == "map":
        n = case["n"]
        st["state"] = gs2d.DeviceMapState.from_tensors(i["delta"], i["t_c"], i["d_c"], i["t_l"])
        st["out"] = gs2d.DeviceSurfels.from_tensors(z(n, 3), z(n, 4), z(n, 2), z(n), z(n, 3))
        st["state_out"] = gs2d.DeviceMapState.from_tensors(z(n, dt=torch.uint8), z(n, dt=torch.int32), z(n),
                                                           z(n, dt=torch.int32))
        st["prm"] = gs2d.StateParams(0.5, 20, 0, -1)
        st["counts"], st["skipped"], st["n_out"] = z(4, dt=torch.int32), z(1, dt=torch.int32), z(1, dt=torch.int32)
        st["keep"], st["new_index"] = z(n, dt=torch.uint8), z(n, dt=torch.int32)
        st["cws"] = _bytes(gs2d.gs2d_map_correct_workspace(N_KF))
        st["kws"] = _bytes(gs2d.gs2d_map_compact_workspace(n))
    elif k == "expand":
        cap = case["w"] * case["h"]
        st["table"] = gs2d.DeviceVoxelTable(1 << 22, 0.02)
        st["out"] = gs2d.DeviceSurfels.from_tensors(z(cap, 3), z(cap, 4), z(cap, 2), z(cap), z(cap, 3))
        st["state"] = gs2d.DeviceMapState(cap, d_c=0.0)
        st["n_new"], st["ws"] = z(1, dt=torch.int32), _bytes(gs2d.gs2d_expand_workspace(st["ccam"]))
        st["prm"] = gs2d.ExpandParams(case["ratio"], 0.99, 0.05, 9, 1)
        st["cap"] = cap
    elif k == "ssim":
        st["g"], st["loss"] = [torch.zeros_like(a) for a in i["ren"]], z(1)
        st["ws"] = _bytes(gs2d.gs2d_mapping_loss_ssim_workspace(st["ccam"]))
    return st


GRADS = ("mu", "quat", "scale", "opacity", "rgb")
IMAGES = ("rgb", "depth", "normal", "opacity")


def run(st):
    case = st["case"]
    k = case["kind"]
    if k == "single":
        r, pose = st["r"], st["pose_t"]
        img = r.forward(st["ds"], pose)
        gs2d.gs2d_mapping_loss(r.rgb, r.depth, r.normal, r.opacity, *st["obs"], r.cam, 0.5, 0.02, *st["g"],
                               st["loss"], st["lws"])
        g = r.backward(st["ds"], pose, *st["g"])
        return dict({n: img[n] for n in IMAGES}, loss=st["loss"], pose6=g["pose6"],
                    **{"d_" + n: g[n] for n in GRADS})
    if k == "track":
        st["cur"].copy_(st["pose_t"])
        gs2d.gs2d_track_step(st["ds"], st["ccam"], st["cfg"], st["prm"], st["cur"], *st["obs"], case["iters"],
                             st["cap"], st["loss"], st["poses"], st["ws"], grad_hist=st["grads"])
        return dict(pose=st["cur"], loss=st["loss"], poses=st["poses"], grads=st["grads"])
    if k == "keyframe":
        r = st["r"]
        r.project(st["ds"], st["pose_t"])
        r.bin_sort(grow=False)
        r.contribution(out=st["contrib"])
        gs2d.gs2d_covisibility(st["contrib"], st["c_kf"], case["n"], 0.5, st["pose_t"], st["kf_t"], 0.9, 0.15,
                               st["counts"], st["score"], st["is_kf"])
        return dict(contrib=st["contrib"], counts=st["counts"], score=st["score"], is_kf=st["is_kf"])
    if k in ("window", "uneven"):
        br = st["br"]
        br.forward(st["ds"], check_status=False)
        gs2d.gs2d_mapping_loss_batch(st["lv"], 0.5, 0.02, st["loss"], st["lws"])
        g = br.backward(st["ds"])
        # a mapping step's results; the images too where they are few
        return dict(loss=st["loss"], grads=[g[n] for n in GRADS], pose6=[b["d_pose6"] for b in br.keep],
                    images=[[b[n] for n in IMAGES] for b in br.keep] if case["views"] <= 8 else [])
    if k == "proposal":
        pr = st["pr"]
        pr.pose.copy_(st["pose_t"][None])
        st["graph"].replay()
        return dict(pose=pr.pose, y=pr.y, proposed=pr.prop, loss_kept=pr.loss_init, loss_proposed=pr.loss_prop,
                    accepted=pr.accepted, x=pr.x)
    if k == "train":
        gs2d.gs2d_net_grad(st["params"], st["x"], st["target"], st["loss"], st["grad"], st["ws"], y=st["y"])
        st["step"] += 1
        gs2d.gs2d_net_adamw(st["params"], st["grad"], st["m"], st["v"], st["step"], lr=1e-4, wd=1e-4)
        return {n: st[n] for n in ("y", "loss", "grad", "params", "m", "v")}
    if k == "forward":
        gs2d.gs2d_net_forward_prepared(st["params"], st["x"], st["y"], st["ws"])
        return dict(y=st["y"])
    if k == "map":
        n, ds, s = case["n"], st["ds"], st["state"]
        gs2d.gs2d_map_observe(st["contrib"], ds.mu, n, st["pose_t"], N_KF, st["prm"], s, st["counts"])
        gs2d.gs2d_map_correct(ds.mu, ds.quat, s.t_c, n, st["old"], st["new"], N_KF, st["cws"], st["skipped"])
        gs2d.gs2d_map_prune(st["contrib"], s.t_c, n, 7, 0.5, st["keep"])
        gs2d.gs2d_map_compact(st["keep"], n, ds, s, st["out"], st["state_out"], st["new_index"], st["n_out"],
                              st["kws"])
        o, so = st["out"], st["state_out"]
        return dict(mu=ds.mu, quat=ds.quat, state=[s.delta, s.t_c, s.d_c, s.t_l], counts=st["counts"],
                    skipped=st["skipped"], new_index=st["new_index"], n_out=st["n_out"],
                    out=[o.mu, o.quat, o.scale, o.opacity, o.rgb], state_out=[so.delta, so.t_c, so.d_c, so.t_l])
    if k == "expand":
        t = st["table"]
        t.clear()
        t.insert(st["act"])
        gs2d.gs2d_expand(st["rgb"], st["depth"], st["ccam"], st["pose_t"], st["u_keep"], st["u_angle"], t, st["prm"],
                         0, st["cap"], st["out"], st["state"], st["n_new"], st["ws"])
        o, s = st["out"], st["state"]
        return dict(n_new=st["n_new"], out=[o.mu, o.quat, o.scale, o.opacity, o.rgb],
                    state=[s.delta, s.t_c, s.d_c, s.t_l])
    gs2d.gs2d_mapping_loss_ssim(*st["ren"], *st["obs"], st["ccam"], 0.125, 0.5, 0.02, *st["g"], st["loss"], st["ws"])
    return dict(loss=st["loss"], g=st["g"])


def work(case):
    k = case["kind"]
    if k in ("train", "forward"):
        B, hw, fl, par = case["batch"], 120 * 160, 0, 0
        shapes = [(60, 80), (30, 40), (15, 20), (8, 10), (4, 5), (2, 3)]
        for l, (h, w) in enumerate(shapes):
            fl += 2 * h * w * 9 * CONV[l] * CONV[l + 1] * (3 if k == "train" and l else 2 if k == "train" else 1)
            par += 9 * CONV[l] * CONV[l + 1] + CONV[l + 1]
        fc = 1536 * 256 + 256 * 6
        fl, par = fl + 2 * fc * (3 if k == "train" else 1), par + fc + 262
        return {"bytes": B * (hw * 16 + 48) + par * (32 if k == "train" else 4), "flops": B * fl}
    if k == "map":
        # contributions, mu, quat and the state in; mu, quat, state, keep, index out; the
        # compacted copy out (scale, opacity and colour in)
        return {"bytes": case["n"] * (4 + 28 + 13 + 28 + 13 + 4 + 24 + 52 + 13), "flops": case["n"] * 70}
    if k == "expand":
        px = case["w"] * case["h"]
        ps = int(px * case["ratio"])
        return {"bytes": px * 8 + ps * (8 + 52 + 13) + case["n"] * 12 + (8 << 22), "flops": ps * 200}
    if k == "ssim":
        return {"bytes": case["w"] * case["h"] * (32 + 16 + 32), "flops": case["w"] * case["h"] * 520}
    if k in ("window", "uneven"):
        px = case["w"] * case["h"] * case["views"] if k == "window" else case["views"] * 400_000
        # images, observations and image gradients; parameters and their gradients
        return {"bytes": px * (32 + 16) + case["n"] * 104, "flops": px * BLENDED * 140}
    w, h = (160, 120) if k == "proposal" else (case["w"], case["h"])
    if k == "keyframe":
        return {"bytes": case["n"] * 60, "flops": w * h * BLENDED * 26}
    if k == "single":
        return {"bytes": case["n"] * 104 + w * h * 48, "flops": w * h * BLENDED * 140}
    if k == "proposal":
        net = work(dict(kind="forward", batch=1))["flops"]
        p = case["passes"]
        return {"bytes": case["n"] * 52 + w * h * 16 + 6_000_000,
                "flops": w * h * BLENDED * 40 * (1 + p) + net * p + 100 * case["n"] * (1 + p)}
    it = case["iters"]
    return {"bytes": case["n"] * 52 + w * h * 16, "flops": it * (w * h * BLENDED * 120 + 100 * case["n"])}


# ---------------------------------------------------------------------------
# the same results in 64 bits, plainly
# ---------------------------------------------------------------------------
ALPHA_MIN, ALPHA_MAX, T_MIN, CUTOFF, NEAR = 1 / 255, 0.99, 1e-4, 9.0, 0.05


def _d(a):
    return a.detach().to(torch.float64)


def _rays(cam):
    f8 = dict(dtype=torch.float64, device=DEV)
    x = (torch.arange(cam.width, **f8) + 0.5 - cam.cx) / cam.fx
    y = (torch.arange(cam.height, **f8) + 0.5 - cam.cy) / cam.fy
    return torch.stack(torch.meshgrid(x, y, indexing="xy") + (torch.ones(cam.height, cam.width, **f8),), -1)


def _columns(quat):
    w, x, y, z = F.normalize(quat, dim=1).unbind(1)
    return (torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + w * z), 2 * (x * z - w * y)], 1),
            torch.stack([2 * (x * y - w * z), 1 - 2 * (x * x + z * z), 2 * (y * z + w * x)], 1),
            torch.stack([2 * (x * z + w * y), 2 * (y * z - w * x), 1 - 2 * (x * x + y * y)], 1))


class _Render64:
    """One view rendered per pixel over conservative tile lists: ray-plane
    intersection, depth order by the centre, alpha blending with the skip,
    clamp, cutoff and stop rules."""

    TILE = 16

    def __init__(self, surf, cam, R, t, tau=None):
        mu, quat, scale, opac, rgb = surf
        self.cam, self.n = cam, mu.shape[0]
        rot = lambda a: a @ R.T
        mc = rot(mu) + t
        axes = [rot(a) for a in _columns(quat)]
        if tau is not None:
            turn = lambda a: torch.linalg.cross(tau[3:].expand_as(a), a)
            mc = mc + tau[:3] + turn(mc)
            axes = [a + turn(a) for a in axes]
        tu, tv, tn = axes
        mu_, mv = scale[:, :1] * tu, scale[:, 1:] * tv
        nn = torch.linalg.cross(mu_, mv)
        n2 = (nn * nn).sum(1, keepdim=True)
        du, dv = torch.linalg.cross(mv, nn) / n2, torch.linalg.cross(nn, mu_) / n2
        dot = lambda a: (a * mc).sum(1, keepdim=True)
        self.Q = torch.cat([nn, dot(nn), du, dot(du), dv, dot(dv), opac[:, None], rgb, tn], 1)
        with torch.no_grad():
            self._lists(mc.detach(), 3.01 * scale.detach().max(1).values)

    def _lists(self, mc, r):
        cam, T = self.cam, self.TILE
        self.tx, self.ty = -(-cam.width // T), -(-cam.height // T)
        z = mc[:, 2]
        far = z - r > 0.02

        def span(a, f, c, n):
            lo = torch.minimum((a - r) / (z - r), (a - r) / (z + r)) * f + c - 1
            hi = torch.maximum((a + r) / (z - r), (a + r) / (z + r)) * f + c + 1
            lo, hi = torch.where(far, lo, 0.0), torch.where(far, hi, float(n))
            return (lo.clamp(0, n) / T).floor().long(), (hi.clamp(-1, n - 1) / T).floor().long()
        x0, x1 = span(mc[:, 0], cam.fx, cam.cx, cam.width)
        y0, y1 = span(mc[:, 1], cam.fy, cam.cy, cam.height)
        cnt = torch.where(z > NEAR, (x1 - x0 + 1).clamp_min(0) * (y1 - y0 + 1).clamp_min(0), 0)
        order = torch.argsort(z, stable=True)
        cnt, nx = cnt[order], (x1 - x0 + 1)[order]
        rank = torch.repeat_interleave(torch.arange(self.n, device=DEV), cnt)
        k = torch.arange(rank.numel(), device=DEV) - (cnt.cumsum(0) - cnt)[rank]
        tile = (y0[order][rank] + k // nx[rank]) * self.tx + x0[order][rank] + k % nx[rank]
        tile, perm = torch.sort(tile, stable=True)
        self.ids = order[rank[perm]]
        self.len = torch.bincount(tile, minlength=self.tx * self.ty)
        self.start = self.len.cumsum(0) - self.len

    def chunks(self):
        by = torch.argsort(self.len, descending=True)
        lens, i = self.len[by].tolist(), 0
        while i < len(lens):
            L = max(lens[i], 1)
            m = max(1, (1 << 25) // (L * self.TILE ** 2))
            yield by[i:i + m], L
            i += m

    def blend(self, Q, tiles, L):
        """(pixel ids, inside flags, list ids, weights [t, p, L], outputs [t, p, 8])."""
        cam, T = self.cam, self.TILE
        p = torch.arange(T * T, device=DEV)
        px = (tiles % self.tx * T)[:, None] + p % T
        py = (tiles // self.tx * T)[:, None] + p // T
        ins = (px < cam.width) & (py < cam.height)
        rx = ((px + 0.5 - cam.cx) / cam.fx).double()[:, :, None]
        ry = ((py + 0.5 - cam.cy) / cam.fy).double()[:, :, None]
        j = torch.arange(L, device=DEV)
        live = j < self.len[tiles][:, None]
        ids = self.ids[torch.where(live, self.start[tiles][:, None] + j, 0)] if self.ids.numel() else \
            torch.zeros(len(tiles), L, dtype=torch.long, device=DEV)
        q = Q.index_select(0, ids.reshape(-1)).reshape(len(tiles), 1, L, 19)
        c = lambda k: q[..., k]
        on = lambda k: c(k) * rx + c(k + 1) * ry + c(k + 2)
        z = c(3) / on(0)
        u, v = z * on(4) - c(7), z * on(8) - c(11)
        rr = u * u + v * v
        with torch.no_grad():
            ok = (rr <= CUTOFF) & (z > NEAR) & live[:, None]
        raw = c(12) * torch.exp(-0.5 * torch.where(ok, rr, 0.0))
        a = raw.clamp_max(ALPHA_MAX)
        a = torch.where(ok & (a >= ALPHA_MIN), a, 0.0)
        after = torch.cumsum(torch.log1p(-a), 2)
        keep = after >= math.log(T_MIN)
        a = torch.where(keep, a, 0.0)
        after = torch.where(keep, after, 0.0)
        before = torch.cat([torch.zeros_like(after[..., :1]), after[..., :-1]], 2)
        w = a * torch.exp(before)
        zz = torch.where(a > 0, z, 0.0)
        out = torch.stack([(w * c(13)).sum(2), (w * c(14)).sum(2), (w * c(15)).sum(2), (w * zz).sum(2),
                           (w * c(16)).sum(2), (w * c(17)).sum(2), (w * c(18)).sum(2), w.sum(2)], 2)
        return (py * cam.width + px), ins, ids, w, out

    def images(self):
        """rgb, depth, normal, opacity, as leaves that take a gradient."""
        img = torch.zeros(self.cam.height * self.cam.width, 8, dtype=torch.float64, device=DEV)
        with torch.no_grad():
            for tiles, L in self.chunks():
                pix, ins, _, _, out = self.blend(self.Q, tiles, L)
                img[pix[ins]] = out[ins]
        h, w = self.cam.height, self.cam.width
        return [a.reshape(s).clone().requires_grad_() for a, s in
                ((img[:, :3], (h, w, 3)), (img[:, 3], (h, w)), (img[:, 4:7], (h, w, 3)), (img[:, 7], (h, w)))]

    def contributions(self):
        total = torch.zeros(self.n, dtype=torch.float64, device=DEV)
        with torch.no_grad():
            for tiles, L in self.chunks():
                _, ins, ids, w, _ = self.blend(self.Q, tiles, L)
                total.index_add_(0, ids.reshape(-1), (w * ins[:, :, None]).sum(1).reshape(-1))
        return total

    def backward(self, images):
        """Carries the images' gradients on to what the view was built from."""
        g = [torch.zeros_like(a) if a.grad is None else a.grad for a in images]
        up = torch.cat([g[0].reshape(-1, 3), g[1].reshape(-1, 1), g[2].reshape(-1, 3), g[3].reshape(-1, 1)], 1)
        Q = self.Q.detach().requires_grad_()
        for tiles, L in self.chunks():
            pix, ins, _, _, out = self.blend(Q, tiles, L)
            (out[ins] * up[pix[ins]]).sum().backward()
        self.Q.backward(Q.grad)


def _pose64(p):
    """Rotation and translation of a pose as the 32-bit numbers a call is given."""
    p = _t(np.concatenate([np.asarray(p.R).reshape(-1), np.asarray(p.t)])).double()
    return p[:9].reshape(3, 3), p[9:]


def _tracking_loss64(img, obs, cam):
    rgb, depth, nrm, op = img
    ok = ((nrm * _rays(cam)).sum(-1) > 0) & (op > 0.95)
    per = (rgb - _d(obs[0])).abs().sum(-1) + (depth / op.clamp_min(1e-6) - _d(obs[1])).abs()
    return (per * ok.detach()).sum() / (cam.width * cam.height)


def _mapping_loss64(img, obs, cam, w_ssim, w_d, w_n):
    rgb, depth, nrm, op = img
    dh = depth / op.clamp_min(1e-6)
    X = dh[..., None] * _rays(cam)
    gx, gy = (X[1:-1, 2:] - X[1:-1, :-2]) / 2, (X[2:, 1:-1] - X[:-2, 1:-1]) / 2
    n = torch.linalg.cross(gx, gy)
    o = op.detach() > 0.5
    ok = o[1:-1, 1:-1] & o[1:-1, 2:] & o[1:-1, :-2] & o[2:, 1:-1] & o[:-2, 1:-1] & ((n.detach() ** 2).sum(-1) > 0)
    n = torch.where(ok[..., None], n, torch.ones_like(n))
    ln = ((1 - (F.normalize(n, dim=-1) * nrm[1:-1, 1:-1]).sum(-1)) * ok).sum()
    total = (1 - w_ssim) * (rgb - _d(obs[0])).abs().sum() + w_d * (dh - _d(obs[1])).abs().sum() + w_n * ln
    if w_ssim:
        k = torch.exp(-torch.arange(-5, 6, dtype=torch.float64, device=DEV) ** 2 / (2 * 1.5 ** 2))
        k = k / k.sum()
        blur = lambda a: F.conv2d(F.conv2d(a, k.reshape(1, 1, 11, 1), padding=(5, 0)), k.reshape(1, 1, 1, 11),
                                  padding=(0, 5))
        x, y = rgb.permute(2, 0, 1)[:, None], _d(obs[0]).permute(2, 0, 1)[:, None]
        mx, my = blur(x), blur(y)
        vx, vy, vxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
        s = (2 * mx * my + 1e-4) * (2 * vxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (vx + vy + 9e-4))
        total = total + w_ssim * (1 - s).sum() / 3
    return total / (cam.width * cam.height)


def _twist64(tau):
    M = torch.zeros(4, 4, dtype=torch.float64, device=DEV)
    M[0, 1], M[0, 2], M[1, 2] = -tau[5], tau[4], -tau[3]
    M[1, 0], M[2, 0], M[2, 1] = tau[5], -tau[4], tau[3]
    M[:3, 3] = tau[:3]
    E = torch.linalg.matrix_exp(M)
    return E[:3, :3], E[:3, 3]


def _net64(params, x):
    """Outputs of the network; x [B, 120, 160, 8]."""
    at, a = 0, x.permute(0, 3, 1, 2)
    for ci, co in zip(CONV[:-1], CONV[1:]):
        W = params[at:at + 9 * ci * co].reshape(co, 3, 3, ci).permute(0, 3, 1, 2)
        at += 9 * ci * co
        a = F.relu(F.conv2d(a, W, params[at:at + co], stride=2, padding=1))
        at += co
    a = a.permute(0, 2, 3, 1).reshape(a.shape[0], -1)
    a = F.relu(F.linear(a, params[at:at + 1536 * 256].reshape(256, 1536), params[at + 1536 * 256:at + 1537 * 256]))
    at += 1537 * 256
    return F.linear(a, params[at:at + 1536].reshape(6, 256), params[at + 1536:at + 1542])


def exact(case, seed):
    k = case["kind"]
    if k in ("window", "uneven"):
        cams, _, sizes = _views(case, seed)
        if sum(c.width * c.height * (m or case["n"]) for c, m in zip(cams, sizes)) > 2e12:
            return None             # over 20 seconds
    i = _inputs(case, seed)
    if k in ("single", "window", "uneven"):
        one = k == "single"
        leaf = [_d(a).requires_grad_() for a in i["surf"]]
        cams, poses = ([i["cam"]], [i["pose"]]) if one else (i["cams"], i["poses"])
        obs, act = ([i["obs"]], [None]) if one else (i["obs"], i["actives"])
        loss, pose6, images = [], [], []
        for c, p, o, a in zip(cams, poses, obs, act):
            tau = torch.zeros(6, dtype=torch.float64, device=DEV, requires_grad=True)
            sub = leaf if a is None else [t[a.long()] for t in leaf]
            r = _Render64(sub, c, *_pose64(p), tau=tau)
            img = r.images()
            L = _mapping_loss64(img, o, c, 0.0, 0.5, 0.02)
            L.backward()
            r.backward(img)
            loss.append(L.detach())
            pose6.append(tau.grad)
            images.append([a.detach() for a in img])
        grads = [a.grad for a in leaf]
        if one:
            return dict(dict(zip(IMAGES, images[0])), loss=loss[0].reshape(1), pose6=pose6[0],
                        **{"d_" + n: g for n, g in zip(GRADS, grads)})
        return dict(loss=torch.stack(loss), grads=grads, pose6=pose6, images=images if case["views"] <= 8 else [])
    if k == "track":
        surf = [_d(a) for a in i["surf"]]
        R, t = _pose64(i["pose"])
        m, v = (torch.zeros(6, dtype=torch.float64, device=DEV) for _ in range(2))
        loss, poses, grads = [], [], []
        for s in range(1, case["iters"] + 1):
            tau = torch.zeros(6, dtype=torch.float64, device=DEV, requires_grad=True)
            r = _Render64(surf, i["cam"], R, t, tau=tau)
            img = r.images()
            L = _tracking_loss64(img, i["obs"], i["cam"])
            L.backward()
            r.backward(img)
            m, v = 0.9 * m + 0.1 * tau.grad, 0.999 * v + 0.001 * tau.grad ** 2
            dR, dt = _twist64(-1e-3 * (m / (1 - 0.9 ** s)) / ((v / (1 - 0.999 ** s)).sqrt() + 1e-8))
            R, t = dR @ R, dR @ t + dt
            loss.append(L.detach())
            poses.append(torch.cat([R.reshape(-1), t]))
            grads.append(tau.grad)
        return dict(pose=poses[-1], loss=torch.stack(loss), poses=torch.stack(poses), grads=torch.stack(grads))
    if k == "keyframe":
        c = _Render64([_d(a) for a in i["surf"]], i["cam"], *_pose64(i["pose"])).contributions()
        a, b = c > 0.5, i["c_kf"] > 0.5
        score = (a & b).sum().double() / (a | b).sum().clamp_min(1)
        return dict(contrib=c, counts=None, score=score.reshape(1), is_kf=None)
    if k == "proposal":
        surf, cam = [_d(a) for a in i["surf"]], i["cam"]
        P = torch.cat([a.reshape(-1) for a in _pose64(i["pose"])])
        look = lambda p: [a.detach() for a in _Render64(surf, cam, p[:9].reshape(3, 3), p[9:]).images()]
        img = look(P)
        kept = _tracking_loss64(img, i["obs"], cam)
        od = _d(i["obs"][1])
        for _ in range(case["passes"]):
            rd = torch.where(img[3] > 0.5, img[1] / img[3].clamp_min(1e-6) - 2.5, 0.0)
            x = torch.cat([img[0], rd[..., None], _d(i["obs"][0]), torch.where(od > 0, od - 2.5, 0.0)[..., None]], 2)
            y = _net64(_d(i["params"]), x[None])
            dR, dt = _twist64(0.03 * y[0])
            prop = torch.cat([(dR @ P[:9].reshape(3, 3)).reshape(-1), dR @ P[9:] + dt])
            pim = look(prop)
            lp = _tracking_loss64(pim, i["obs"], cam)
            was = kept
            if lp <= kept:
                P, img, kept = prop, pim, lp
        return dict(pose=P[None], y=y, proposed=prop[None], loss_kept=was.reshape(1), loss_proposed=lp.reshape(1),
                    accepted=None, x=x[None])
    if k == "forward":
        return dict(y=_net64(_d(i["params"]), _d(i["x"])))
    if k == "train":
        p = _d(i["params"]).requires_grad_()
        y = _net64(p, _d(i["x"]))
        L = 0.5 * ((y - _d(i["target"])) ** 2).sum() / case["batch"]
        L.backward()
        g = p.grad
        m, v = 0.9 * _d(i["m"]) + 0.1 * g, 0.999 * _d(i["v"]) + 0.001 * g * g
        step = (m / (1 - 0.9 ** 101)) / ((v / (1 - 0.999 ** 101)).sqrt() + 1e-8)
        return dict(y=y.detach(), loss=L.detach().reshape(1), grad=g, params=p.detach() * (1 - 1e-8) - 1e-4 * step,
                    m=m, v=v)
    if k == "map":
        R, t = _pose64(i["pose"])
        mu, quat = _d(i["surf"][0]), _d(i["surf"][1])
        dist = (mu + R.T @ t).norm(dim=1)
        closer = (i["delta"] > 0) & (i["contrib"] > 0.5) & (dist < _d(i["d_c"]))
        d_c = torch.where(closer, dist, _d(i["d_c"]))
        t_c = torch.where(closer, N_KF, i["t_c"].long())
        A, B = _d(i["old"]), _d(i["new"])
        Ro, to, Rn, tn = A[:, :9].reshape(-1, 3, 3), A[:, 9:], B[:, :9].reshape(-1, 3, 3), B[:, 9:]
        dR = Rn.transpose(1, 2) @ Ro
        dt = (Rn.transpose(1, 2) @ (to - tn)[:, :, None])[:, :, 0]
        w = 0.5 * (1 + dR.diagonal(dim1=1, dim2=2).sum(1)).clamp_min(0).sqrt()
        axis = torch.stack([dR[:, 2, 1] - dR[:, 1, 2], dR[:, 0, 2] - dR[:, 2, 0], dR[:, 1, 0] - dR[:, 0, 1]], 1)
        dq = torch.cat([w[:, None], axis / (4 * w[:, None])], 1)
        j, on = t_c.clamp_max(N_KF - 1), (t_c < N_KF)[:, None]
        mu = torch.where(on, (dR[j] @ mu[:, :, None])[:, :, 0] + dt[j], mu)
        a, q = dq[j], quat
        turned = torch.stack([a[:, 0] * q[:, 0] - a[:, 1] * q[:, 1] - a[:, 2] * q[:, 2] - a[:, 3] * q[:, 3],
                              a[:, 0] * q[:, 1] + a[:, 1] * q[:, 0] + a[:, 2] * q[:, 3] - a[:, 3] * q[:, 2],
                              a[:, 0] * q[:, 2] - a[:, 1] * q[:, 3] + a[:, 2] * q[:, 0] + a[:, 3] * q[:, 1],
                              a[:, 0] * q[:, 3] + a[:, 1] * q[:, 2] - a[:, 2] * q[:, 1] + a[:, 3] * q[:, 0]], 1)
        quat = torch.where(on, turned, quat)
        keep = ~((t_c == 7) & (i["contrib"] < 0.5))

        def packed(x):
            o = torch.zeros_like(x)
            o[:int(keep.sum())] = x[keep]
            return o
        return dict(mu=mu, quat=quat, state=[None, None, d_c, None], counts=None, skipped=None, new_index=None,
                    n_out=None, out=[packed(a) for a in (mu, quat, *(_d(a) for a in i["surf"][2:]))],
                    state_out=[None, None, packed(d_c), None])
    if k == "expand":
        cam, (R, t) = i["cam"], _pose64(i["pose"])
        D = _d(i["depth"])
        Xc = D[..., None] * _rays(cam)
        ok = D > 0
        gx, gy = (Xc[1:-1, 2:] - Xc[1:-1, :-2]) / 2, (Xc[2:, 1:-1] - Xc[:-2, 1:-1]) / 2
        c = torch.linalg.cross(gx, gy)
        inner = ok[1:-1, 1:-1] & ok[1:-1, 2:] & ok[1:-1, :-2] & ok[2:, 1:-1] & ok[:-2, 1:-1] & ((c * c).sum(-1) > 0)
        N = F.pad(F.normalize(c, dim=-1), (0, 0, 1, 1, 1, 1)).reshape(-1, 3)
        has = F.pad(inner, (1, 1, 1, 1)).reshape(-1)
        pix = (ok & (i["u_keep"] < np.float32(case["ratio"]))).reshape(-1).nonzero()[:, 0]
        Xk = Xc.reshape(-1, 3)[pix]
        Xw = (Xk - t) @ R
        key = lambda x: ((x.float() * 50.0).floor().long() * _t([1, 1 << 20, 1 << 40], torch.long)).sum(1)
        new = has[pix] & ~torch.isin(key(Xw), key(i["act"]))
        near = []
        for s in range(0, len(pix), 2048):
            d = (Xw[s:s + 2048, None] - Xw[None]).norm(dim=2)
            d[torch.arange(d.shape[0]), torch.arange(s, s + d.shape[0])] = math.inf
            near.append(d.min(1).values)
        near = torch.cat(near)[new]
        near = torch.where(near.isfinite(), near, 0.05)
        # the tangent frame's quaternion has either sign: no one value
        rows = lambda x, *s: torch.cat([x, torch.zeros(cam.width * cam.height - len(x), *s, dtype=x.dtype, device=DEV)])
        return dict(n_new=None, out=[rows(Xw[new], 3), None, rows(torch.stack([near, near], 1), 2),
                                     rows(torch.full_like(near, 0.99)), rows(_d(i["rgb"]).reshape(-1, 3)[pix[new]], 3)],
                    state=[None, None, rows(Xk[new].norm(dim=1)), None])
    ren = [_d(a).requires_grad_() for a in i["ren"]]
    L = _mapping_loss64(ren, i["obs"], i["cam"], 0.125, 0.5, 0.02)
    L.backward()
    return dict(loss=L.detach().reshape(1), g=[a.grad for a in ren])
