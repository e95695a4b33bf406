"""GPU parity of the voxel table and of gs2d_expand (Sec. III-E) against the
FP64 oracle ``oracle.expand``.

Decisions are compared exactly where they are unique: the GPU forms voxel
coordinates as floor(X / r_h) in FP32, so a point within 1e-4 r_h of a voxel
face may land on either side; such points are left out of the exact
comparison (both outcomes are valid).  Everything else -- which pixels enter
P_s, which points become surfels, their order, colours and states -- is
bit-exact; positions, scales (nearest-neighbour distances), frames and
viewpoint distances are within 1e-5 relative (FP32 of a few operations).
"""
import numpy as np
import pytest

import oracle.expand as ex
import oracle.map_state as ms
from paper_2506_00970_gb300 import scenes
from gpu_helpers import to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_00970_gb300 import gs2d
    gs2d.lib()
    return torch


def _near_face(X, voxel, tol=1e-4):
    f = np.asarray(X, np.float64) / voxel
    return (np.abs(f - np.round(f)) < tol).any(-1)


def test_voxel_table_insert_query(torch_cuda):
    torch = torch_cuda
    from paper_2506_00970_gb300 import gs2d
    rng = np.random.default_rng(0)
    vox = 0.05
    a = rng.uniform(-3, 3, (20000, 3)).astype(np.float32)
    a = a[~_near_face(a, vox)]                   # inserted voxels are unambiguous
    b = np.concatenate([a[:5000] + rng.uniform(-0.01, 0.01, (5000, 3)).astype(np.float32),
                        rng.uniform(-3, 3, (20000, 3)).astype(np.float32)])
    t = gs2d.DeviceVoxelTable(1 << 16, vox)
    T = lambda x: torch.tensor(x, device="cuda")
    mask = (rng.uniform(size=len(a)) < 0.7).astype(np.uint8)
    t.insert(T(a), T(mask))
    occ = t.query(T(b)).cpu().numpy().astype(bool)
    torch.cuda.synchronize()
    assert int(t.status.item()) == 0
    occupied = {tuple(v) for v in ex.voxel_index(a[mask.astype(bool)], vox)}
    expect = np.array([tuple(v) in occupied for v in ex.voxel_index(b, vox)])
    ok = ~_near_face(b, vox)
    assert np.array_equal(occ[ok], expect[ok])
    assert occ.sum() > 1500
    # a full table reports it and returns (every probe loop is bounded)
    small = gs2d.DeviceVoxelTable(64, vox)
    small.insert(T(a))
    torch.cuda.synchronize()
    assert int(small.status.item()) == 3
    small.clear()
    torch.cuda.synchronize()
    assert int(small.status.item()) == 0 and not bool(small.query(T(a[:10])).any())


def _run_expand(torch, rgb, depth, cam, pose, u_keep, u_angle, ratio, kf, table=None, n_map=0,
                capacity=None, insert=0, max_scale=0.05):
    from paper_2506_00970_gb300 import gs2d
    T = lambda x: torch.tensor(np.ascontiguousarray(x), device="cuda")
    H, W = depth.shape
    cap = capacity if capacity is not None else n_map + H * W
    f = dict(dtype=torch.float32, device="cuda")
    out = gs2d.DeviceSurfels.from_tensors(torch.full((cap, 3), -1.0, **f),
                                          torch.full((cap, 4), -1.0, **f),
                                          torch.full((cap, 2), -1.0, **f),
                                          torch.full((cap,), -1.0, **f),
                                          torch.full((cap, 3), -1.0, **f))
    st = gs2d.DeviceMapState(cap, kf_id=-5, d_c=-1.0, active=False)
    n_new = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    ccam = gs2d.camera(cam)
    ws = torch.empty(gs2d.gs2d_expand_workspace(ccam), dtype=torch.uint8, device="cuda")
    prm = gs2d.ExpandParams(ratio, 0.99, max_scale, kf, insert)
    p12 = np.concatenate([pose.R.reshape(-1), pose.t]).astype(np.float32)
    gs2d.gs2d_expand(T(rgb), T(depth), ccam, T(p12), T(u_keep), T(u_angle), table, prm, n_map,
                     cap, out, st, n_new, ws)
    torch.cuda.synchronize()
    return out, st, int(n_new.item())


@pytest.mark.parametrize("w,h,ratio,table", [(160, 120, 0.3, False), (640, 480, 0.08, True),
                                             (1200, 680, 0.04, True)])
def test_expand_matches_oracle(torch_cuda, w, h, ratio, table):
    torch = torch_cuda
    from paper_2506_00970_gb300 import gs2d
    f = {160: 150.0, 640: 525.0, 1200: 600.0}[w]
    cam = scenes.Camera(f, f, w / 2, h / 2, w, h)
    rgb, depth = scenes.rgbd_frame(w, cam)
    rng = np.random.default_rng(w)
    u_keep = rng.uniform(size=(h, w)).astype(np.float32)
    u_angle = rng.uniform(size=(h, w)).astype(np.float32)
    pose = scenes.perturb_pose(scenes.identity_pose(), 0.3, 20.0, seed=w)
    R = pose.R.astype(np.float32).astype(np.float64)
    t = pose.t.astype(np.float32).astype(np.float64)
    vox = 0.04
    occ_pts = np.zeros((0, 3), np.float32)
    tb = None
    if table:
        # the active map: world points of a quarter of the frame's P_s
        pre = ex.expand(rgb, depth, cam, R, t, u_keep, u_angle, ratio, 0)
        occ_pts = pre["ps_world"][::4].astype(np.float32)
        tb = gs2d.DeviceVoxelTable(1 << 18, vox)
        tb.insert(torch.tensor(occ_pts, device="cuda"))
    o = ex.expand(rgb, depth, cam, R, t, u_keep, u_angle, ratio, 7,
                  occupied={tuple(v) for v in ex.voxel_index(occ_pts, vox)}, voxel=vox)
    out, st, k = _run_expand(torch, rgb, depth, cam, pose, u_keep, u_angle, ratio, 7, tb)
    # ambiguous voxel decisions: a P_s point or an occupying point near a face
    amb_pix = set()
    if table:
        near = _near_face(o["ps_world"], vox)
        occ_near = {tuple(v) for v in ex.voxel_index(occ_pts[_near_face(occ_pts, vox)], vox)}
        for j, p in enumerate(o["ps_pixel"]):
            if near[j] or tuple(o["ps_voxel"][j]) in occ_near:
                amb_pix.add(int(p))
    g_mu = to_np(out.mu[:k])
    # match GPU surfels to pixels through their positions' order: both are in pixel order
    o_pix = o["pixel"]
    assert abs(k - len(o_pix)) <= len(amb_pix)
    if not amb_pix:
        assert k == len(o_pix)
    # align by pixel: recover the GPU pixel of each surfel from its colour row
    # and position is not needed -- both lists are stable in pixel order, so
    # drop ambiguous pixels from the oracle list and compare against the GPU
    # entries whose positions match
    keep_o = np.array([int(p) not in amb_pix for p in o_pix], bool)
    # GPU entries: the same filter needs the GPU pixel; project back the GPU
    # centre to the image (exact pixel centre up to FP32)
    Xc = g_mu @ R.T + t
    gp = np.round(Xc[:, 1] / Xc[:, 2] * cam.fy + cam.cy - 0.5).astype(int) * w + \
        np.round(Xc[:, 0] / Xc[:, 2] * cam.fx + cam.cx - 0.5).astype(int)
    keep_g = np.array([int(p) not in amb_pix for p in gp], bool)
    assert np.array_equal(gp[keep_g], o_pix[keep_o])
    sel = keep_g
    np.testing.assert_allclose(g_mu[sel], o["mu"][keep_o], rtol=1e-5, atol=1e-5)
    np.testing.assert_allclose(to_np(out.scale[:k])[sel], o["scale"][keep_o], rtol=1e-4)
    np.testing.assert_array_equal(to_np(out.rgb[:k])[sel], o["rgb"][keep_o].astype(np.float32))
    np.testing.assert_allclose(to_np(out.opacity[:k]), np.float32(0.99))
    Rg = ms.quat_matrix(to_np(out.quat[:k]))[sel]
    Ro = o["R"][keep_o]
    np.testing.assert_allclose(Rg[:, :, 2], Ro[:, :, 2], atol=2e-4)      # the normal
    # the tangent basis switches branch with the sign of n_z: compare the
    # random tangents where that sign is unambiguous, check the rest is a frame
    uni = np.abs(Ro[:, 2, 2]) > 1e-4
    np.testing.assert_allclose(Rg[uni], Ro[uni], atol=2e-4)
    np.testing.assert_allclose(np.einsum("kij,kil->kjl", Rg, Rg), np.tile(np.eye(3), (len(Rg), 1, 1)),
                               atol=1e-5)
    np.testing.assert_allclose(np.linalg.norm(to_np(out.quat[:k]), axis=1), 1.0, atol=1e-5)
    assert np.all(st.delta[:k].cpu().numpy() == 1) and np.all(st.t_c[:k].cpu().numpy() == 7)
    assert np.all(st.t_l[:k].cpu().numpy() == 7)
    np.testing.assert_allclose(to_np(st.d_c[:k])[sel], o["d_c"][keep_o], rtol=1e-5)
    # nothing written past the new surfels
    assert bool((out.mu[k:] == -1.0).all())


def test_expand_capacity_insert_and_edge_cases(torch_cuda):
    torch = torch_cuda
    from paper_2506_00970_gb300 import gs2d
    cam = scenes.Camera(150.0, 150.0, 80.0, 60.0, 160, 120)
    rgb, depth = scenes.rgbd_frame(11, cam)
    rng = np.random.default_rng(11)
    u_keep = rng.uniform(size=depth.shape).astype(np.float32)
    u_angle = rng.uniform(size=depth.shape).astype(np.float32)
    pose = scenes.identity_pose()
    # appended after an existing map of 100 surfels
    out, st, k = _run_expand(torch, rgb, depth, cam, pose, u_keep, u_angle, 0.2, 3, n_map=100)
    assert k > 100 and bool((out.mu[:100] == -1.0).all()) and bool((out.mu[100:100 + k] != -1).any())
    # too small a capacity: nothing written, the count still reported, status set
    tb = gs2d.DeviceVoxelTable(1 << 14, 0.05)
    out2, _, k2 = _run_expand(torch, rgb, depth, cam, pose, u_keep, u_angle, 0.2, 3, table=tb,
                              capacity=k - 1)
    assert k2 == k and int(tb.status.item()) == 3 and bool((out2.mu == -1.0).all())
    # with insert_new, the same frame a second time adds nothing
    tb.clear()
    _, _, k3 = _run_expand(torch, rgb, depth, cam, pose, u_keep, u_angle, 0.2, 3, table=tb,
                           insert=1)
    _, _, k4 = _run_expand(torch, rgb, depth, cam, pose, u_keep, u_angle, 0.2, 3, table=tb,
                           insert=1)
    assert k3 == k and k4 == 0
    # an empty frame and a frame with a single valid pixel
    z = np.zeros_like(depth)
    _, _, k5 = _run_expand(torch, rgb, z, cam, pose, u_keep, u_angle, 1.0, 0)
    assert k5 == 0
    one = np.zeros_like(depth)
    one[50:53, 60:63] = 1.0                      # only the centre pixel has a normal
    u1 = np.ones_like(u_keep)
    u1[51, 61] = 0.0                             # and only it is kept
    out6, _, k6 = _run_expand(torch, rgb, one, cam, pose, u1, u_angle, 0.5, 0, max_scale=0.07)
    assert k6 == 1
    np.testing.assert_allclose(to_np(out6.scale[:1]), 0.07)   # no neighbour in P_s


@pytest.mark.parametrize("w,h,ratio,f,cx,outliers", [
    (61, 47, 1.0, 60.0, 30.5, 0.0),          # every pixel a point
    (333, 251, 0.3, 300.0, 166.5, 0.01),     # depth outliers: neighbours far from the pixel
    (333, 251, 0.003, 300.0, 400.0, 0.05),   # sparse points, principal point off the image
    (333, 251, 0.04, 90.0, 166.5, 0.0),      # wide field of view
    (2100, 2003, 0.01, 1500.0, 1050.0, 0.0)  # more pixel blocks than sum their counts themselves
])
def test_expand_nearest_is_the_minimum(torch_cuda, w, h, ratio, f, cx, outliers):
    """The windowed neighbour search against the k-d tree over all of P_s;
    the bound is the rounding of two FP32 points (8 operations each, at the
    scale of the camera-space point plus the translation)."""
    torch = torch_cuda
    cam = scenes.Camera(f, f, cx, h / 2, w, h)
    rgb, depth = scenes.rgbd_frame(w + h, cam)
    rng = np.random.default_rng(w)
    depth = np.where(rng.uniform(size=depth.shape) < outliers, 6.0 * depth, depth).astype(np.float32)
    u_keep = rng.uniform(size=(h, w)).astype(np.float32)
    u_angle = rng.uniform(size=(h, w)).astype(np.float32)
    pose = scenes.perturb_pose(scenes.identity_pose(), 0.3, 20.0, seed=w)
    R = pose.R.astype(np.float32).astype(np.float64)
    t = pose.t.astype(np.float32).astype(np.float64)
    o = ex.expand(rgb, depth, cam, R, t, u_keep, u_angle, ratio, 0)
    out, _, k = _run_expand(torch, rgb, depth, cam, pose, u_keep, u_angle, ratio, 0)
    assert k == len(o["pixel"])
    size = np.linalg.norm(o["mu"] @ R.T + t, axis=1) + np.abs(t).sum()
    tol = 32 * 2.0 ** -24 * size + 1e-6 * o["scale"][:, 0]
    err = np.abs(to_np(out.scale[:k])[:, 0] - o["scale"][:, 0])
    assert np.all(err <= tol), (err / tol).max()
