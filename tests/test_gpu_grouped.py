"""The grouped one-pixel compositing loops (four (pixel, surfel) evaluations
in flight per thread, chosen for tile grids too small to fill the GPU)
against the plain loops: the same evaluations blended in the same order, so
forward images, compositing state and whole tracking frames are
bit-identical whichever form runs."""
import numpy as np
import pytest

from paper_2506_00970_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_00970_gb300 import gs2d
    gs2d.lib()
    yield torch
    gs2d.gs2d_set_grouped_tiles(-1)


def _forward(gs2d, ds, cam, pose, grouped):
    gs2d.gs2d_set_grouped_tiles(1 << 30 if grouped else 0)
    r = gs2d.Rasterizer(cam, ds.n)
    out = r.forward(ds, gs2d.pose_tensor(pose))
    return {k: v.detach().cpu().numpy() for k, v in out.items()}


CASES = [
    # (scene, camera, pose): the c1-style slab, a small room view, a dense
    # low-resolution view of a large room (long tile lists), a ragged image
    ("slab", scenes.Camera(150.0, 150.0, 80.0, 60.0, 160, 120), None),
    ("room30k", scenes.Camera(262.5, 262.5, 160.0, 120.0, 320, 240), 3),
    ("room200k", scenes.Camera(150.0, 150.0, 80.0, 60.0, 160, 120), 100),
    ("room30k", scenes.Camera(200.0, 210.0, 97.0, 53.5, 197, 109), 5),
]


def _scene(name, seed):
    if name == "slab":
        return scenes.slab_scene(0, 4096), scenes.identity_pose()
    n = 30_000 if name == "room30k" else 200_000
    return scenes.room_scene(0, n), scenes.room_pose(seed)


@pytest.mark.parametrize("case", range(len(CASES)))
def test_grouped_forward_is_bit_identical(torch_cuda, case):
    from paper_2506_00970_gb300 import gs2d
    name, cam, seed = CASES[case]
    s, pose = _scene(name, seed)
    ds = gs2d.DeviceSurfels(s)
    a = _forward(gs2d, ds, cam, pose, grouped=False)
    b = _forward(gs2d, ds, cam, pose, grouped=True)
    gs2d.gs2d_set_grouped_tiles(-1)
    assert a["opacity"].max() > 0.5
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


@pytest.mark.parametrize("case", [1, 2, 3])
def test_grouped_tracking_frame_is_bit_identical(torch_cuda, case):
    """20 fused tracking iterations (forward, loss, pose backward, AdamW,
    retraction) give the same loss and pose histories in both forms."""
    torch = torch_cuda
    from paper_2506_00970_gb300 import gs2d
    name, cam, seed = CASES[case]
    s, gt = _scene(name, seed)
    ds = gs2d.DeviceSurfels(s)
    img = _forward(gs2d, ds, cam, gt, grouped=False)
    obs_rgb = torch.tensor(img["rgb"], device="cuda")
    obs_d = torch.tensor(img["depth"] / np.maximum(img["opacity"], 1e-6), device="cuda")
    start = gs2d.pose_tensor(scenes.perturb_pose(gt, 0.02, 1.0, seed=7))
    ccam, cfg = gs2d.camera(cam), gs2d.default_config()
    prm = gs2d.default_track_params(stop_tol=0.0)
    cap = 8 * s.n
    hist = []
    for grouped in (False, True):
        gs2d.gs2d_set_grouped_tiles(1 << 30 if grouped else 0)
        ws = torch.empty(gs2d.gs2d_track_workspace(s.n, cap, ccam, cfg), dtype=torch.uint8,
                         device="cuda")
        pose = start.clone()
        lh = torch.zeros(20, device="cuda")
        ph = torch.zeros(20, 12, device="cuda")
        gs2d.gs2d_track_step(ds, ccam, cfg, prm, pose, obs_rgb, obs_d, 20, cap, lh, ph, ws)
        torch.cuda.synchronize()
        assert int(gs2d.gs2d_track_status(ws).item()) == 0
        hist.append((lh.cpu().numpy(), ph.cpu().numpy(), pose.cpu().numpy()))
    gs2d.gs2d_set_grouped_tiles(-1)
    assert hist[0][0][0] > 0
    for x, y in zip(hist[0], hist[1]):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("w,h,f,tile", [
    (160, 120, 150.0, (16, 16)),     # lists of a few batches
    (112, 84, 105.0, (16, 16)),      # quadrants of more than 768 keys
    (64, 48, 60.0, (16, 16)),        # segments too long for the quadrant form
    (101, 77, 95.0, (8, 32)),        # the other tile shapes, ragged image
    (101, 77, 95.0, (32, 8)),
    (333, 251, 275.0, (16, 16)),     # more tiles than may split, some of them long
])
def test_grouped_forms_agree_over_list_lengths_and_shapes(torch_cuda, w, h, f, tile):
    """Forward images and a short tracking call, whole tiles against quadrants
    and against the library's choice per tile: bit-identical."""
    torch = torch_cuda
    from paper_2506_00970_gb300 import gs2d
    cam = scenes.Camera(f, f, w / 2, h / 2, w, h)
    s = scenes.room_scene(3, 200_000)
    ds = gs2d.DeviceSurfels(s)
    gt = scenes.room_pose(11)
    ccam, cfg = gs2d.camera(cam), gs2d.default_config(tile)
    prm = gs2d.default_track_params(stop_tol=0.0)
    cap = 8 * s.n
    obs, res = None, []
    for limit in (0, 1 << 30, -1):
        gs2d.gs2d_set_grouped_tiles(limit)
        r = gs2d.Rasterizer(cam, s.n, tile=tile)
        out = {k: v.clone() for k, v in r.forward(ds, gs2d.pose_tensor(gt)).items()}
        if obs is None:
            obs = out["rgb"], out["depth"] / out["opacity"].clamp_min(1e-6)
        ws = torch.empty(gs2d.gs2d_track_workspace(s.n, cap, ccam, cfg), dtype=torch.uint8,
                         device="cuda")
        pose = gs2d.pose_tensor(scenes.perturb_pose(gt, 0.02, 1.0, seed=7))
        lh, gh = torch.zeros(4, device="cuda"), torch.zeros(4, 6, device="cuda")
        gs2d.gs2d_track_step(ds, ccam, cfg, prm, pose, *obs, 4, cap, lh, None, ws, grad_hist=gh)
        torch.cuda.synchronize()
        assert int(gs2d.gs2d_track_status(ws).item()) == 0
        res.append(dict(out, loss=lh, grad=gh, pose=pose))
    gs2d.gs2d_set_grouped_tiles(-1)
    assert float(res[0]["loss"][0]) > 0
    for other in res[1:]:
        for k in res[0]:
            assert torch.equal(res[0][k], other[k]), k


@pytest.mark.parametrize("w,h,f", [
    (160, 120, 150.0),     # every tile may split
    (101, 77, 95.0),       # ragged image, the last row of tiles one pixel high
    (333, 251, 275.0),     # more tiles than may split
])
def test_tiles_four_pixels_high_have_quadrants_of_their_own(torch_cuda, w, h, f):
    """A 64x4 tile has no 8 x 8 quadrants: its quadrants are 16 x 4.  The forms
    agree bit for bit, and the images equal the 16x16 tiles' but for the point
    at which intersections are re-based."""
    from gpu_helpers import assert_images_close
    from paper_2506_00970_gb300 import gs2d
    test_grouped_forms_agree_over_list_lengths_and_shapes(torch_cuda, w, h, f, (64, 4))
    s, pose = scenes.room_scene(3, 30_000), gs2d.pose_tensor(scenes.room_pose(11))
    ds, cam, out = gs2d.DeviceSurfels(s), scenes.Camera(f, f, w / 2, h / 2, w, h), []
    for tile in ((16, 16), (64, 4)):
        img = gs2d.Rasterizer(cam, s.n, tile=tile).forward(ds, pose)
        out.append({k: v.cpu().numpy() for k, v in img.items()})
    assert out[0]["opacity"].max() > 0.9
    assert_images_close(out[1], {k: out[0][k].astype(np.float64)
                                 for k in ("rgb", "depth", "normal", "opacity")})


@pytest.mark.parametrize("w,h,f", [(160, 120, 150.0), (333, 251, 275.0)])
@pytest.mark.parametrize("past", [0, 1])
def test_tracking_forms_agree_at_the_line_between_their_launches(torch_cuda, w, h, f, past):
    """The last map size that runs whole tiles only, and the first whose tiles
    may split (8,000 surfels and 30 a tile); lists of up to 256 keys, which are
    ordered by rank, and longer ones: bit-identical histories in every form."""
    torch = torch_cuda
    from paper_2506_00970_gb300 import gs2d
    cam = scenes.Camera(f, f, w / 2, h / 2, w, h)
    n_tiles = -(-w // 16) * -(-h // 16)
    s = scenes.room_scene(4, 8000 + 30 * n_tiles + past)
    ds, gt = gs2d.DeviceSurfels(s), scenes.room_pose(11)
    img = gs2d.Rasterizer(cam, s.n).forward(ds, gs2d.pose_tensor(gt))
    obs = img["rgb"].clone(), img["depth"] / img["opacity"].clamp_min(1e-6)
    ccam, cfg, cap = gs2d.camera(cam), gs2d.default_config(), 8 * s.n
    res = []
    for limit in (0, 1 << 30, -1):
        gs2d.gs2d_set_grouped_tiles(limit)
        ws = torch.empty(gs2d.gs2d_track_workspace(s.n, cap, ccam, cfg), dtype=torch.uint8, device="cuda")
        pose = gs2d.pose_tensor(scenes.perturb_pose(gt, 0.02, 1.0, seed=7))
        lh, gh = torch.zeros(4, device="cuda"), torch.zeros(4, 6, device="cuda")
        gs2d.gs2d_track_step(ds, ccam, cfg, gs2d.default_track_params(stop_tol=0.0), pose, *obs, 4, cap,
                             lh, None, ws, grad_hist=gh)
        torch.cuda.synchronize()
        assert int(gs2d.gs2d_track_status(ws).item()) == 0
        res.append((lh, gh, pose))
    gs2d.gs2d_set_grouped_tiles(-1)
    assert float(res[0][0][0]) > 0
    for other in res[1:]:
        for a, b in zip(res[0], other):
            assert torch.equal(a, b)
