"""Sample counts of the FP32 render's forms where many rays pass the termination
threshold within the rounding of their products: every form counts as the
packed queue does, and counting costs little."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2404_09531_gb300 as om
from _util import gpu_scene

pytestmark = pytest.mark.gpu


def _camera(width, height):
    cam = synth.make_cameras(1)[0]
    f = np.float32(float(cam["fy"]) * height / float(cam["height"]))
    return dict(cam, width=width, height=height, fx=f, fy=f, cx=np.float32(0.5 * width), cy=np.float32(0.5 * height))


def _fog(sigma, holes=False, brick=0):
    """Fog of about the optical depth sigma per sample in the whole box (or in
    four of five occupancy cells, of different heights)."""
    spec = synth.scene_spec(1, step=1.0 / 4096, n_max=2048)
    sc = synth.make_scene(spec)
    rng = np.random.default_rng(3)
    sc["grid"][..., 0] = (np.log(sigma * 4096) + 0.1 * rng.normal(size=sc["grid"].shape[:3])).astype(np.float32)
    for k in ("p_xy", "p_xz", "p_yz"):
        sc[k][..., 0] = 0.0
    sc["occ"] = np.full_like(sc["occ"], 0.12) * np.array([-1.0, 1.0], np.float32)
    if holes:
        sc["occ"][..., 1] = rng.uniform(-0.1, 0.12, sc["occ"].shape[:2])
        sc["occ"][rng.uniform(size=sc["occ"].shape[:2]) < 0.2] = (1.0, -1.0)
    if brick:
        table = oracle.brick_table(synth.scene_spec(1, step=1.0 / 4096, n_max=2048, brick=brick), sc["occ"])
        pool = oracle.extract_bricks(spec.L, brick, table, sc["grid"])
        sc = dict(sc, spec=synth.scene_spec(1, step=1.0 / 4096, n_max=2048, brick=brick), grid=pool, table=table)
    return sc


def _tiles(rays, w, h):
    """The image's rays in 8 x 4 tiles of 32, the places outside the image filled
    with rays that miss the box, and the order that takes the tiles' values back."""
    W, H = (w + 7) // 8 * 8, (h + 3) // 4 * 4
    full = np.tile(np.array([0, 0, 9, 0, 0, 1], np.float32), (H, W, 1))
    full[:h, :w] = rays.reshape(h, w, 6)
    order = np.arange(H * W).reshape(H // 4, 4, W // 8, 8).transpose(0, 2, 1, 3).reshape(-1)
    back = np.empty_like(order)
    back[order] = np.arange(H * W)
    return torch.as_tensor(full.reshape(-1, 6)[order]).cuda(), torch.as_tensor(back.reshape(H, W)[:h, :w].reshape(-1)).cuda()


@pytest.mark.parametrize("sigma,thr,holes,brick", [(0.012, 1e-4, False, 0), (0.05, 1e-3, True, 0), (0.3, 0.05, False, 8),
                                                   (0.004, 0.3, True, 8), (0.002, 0.05, False, 0)])
def test_counts_in_fog(sigma, thr, holes, brick):
    w, h = 203, 85  # ragged tiles; more than 2^14 rays
    scene = gpu_scene(_fog(sigma, holes, brick), t_thr=thr)
    cam = _camera(w, h)
    tiled, back = _tiles(oracle.camera_rays(cam), w, h)
    assert tiled.shape[0] >= 1 << 14
    _, queue = om.render(scene, rays=tiled)
    want = queue[back]
    # the saved training state: transmittances that rounding brought just below the threshold
    _, saved, _ = om.train_fwd(scene, tiled, torch.zeros(tiled.shape[0], 3, device="cuda"))
    state = saved.view(-1, 20)
    cnt = state[:, 8].contiguous().view(torch.int32)
    assert torch.equal(cnt, queue)
    near = (state[:, 7] < thr) & (state[:, 7] > thr * (1 - 1e-6 - 1.3e-7 * cnt))
    if sigma < 0.05:
        assert int(near.sum()) >= 20
    rgb, got = om.render(scene, camera=cam)
    assert torch.equal(got, want)
    for fill in (_camera(512, 256), _camera(1024, 1024)):
        g_rgb, g = om.render_cameras(scene, [cam, fill])
        assert torch.equal(g[: w * h], want) and torch.equal(g_rgb[: w * h], rgb)
    for n in (1, 15, 16, 17, 31, 33, 4999):
        at = 32 * int(near.nonzero()[0, 0] // 32) if near.any() else 0
        part = tiled[at:at + n].contiguous()
        _, got = om.render(scene, rays=part)
        assert torch.equal(got, queue[at:at + n])


def test_counting_costs_little_in_fog():
    """One ray of forty is counted again: a frame with counts takes less than
    twice the time of the pixels alone."""
    scene = gpu_scene(_fog(0.012))
    cam = _camera(1280, 720)

    def fastest(count):
        times = []
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            om.render(scene, camera=cam, want_count=count)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    assert fastest(True) <= 2 * fastest(False)


def test_counts_of_opaque_samples_in_ramps():
    """Occupancy ramps over most of the box and opacities near 1, where a factor
    rounded another way would move the transmittance most: thresholds at the
    queue's own transmittances after two samples, and one step beside them."""
    sc = synth.make_scene(1)
    sc["grid"][..., 0] = np.random.default_rng(5).uniform(np.log(256 * 0.5), np.log(256 * 12), sc["grid"].shape[:3])
    for k in ("p_xy", "p_xz", "p_yz"):
        sc[k][..., 0] = 0.0
    sc["occ"] = np.full_like(sc["occ"], 0.12) * np.array([-1.0, 1.0], np.float32)
    rng = np.random.default_rng(6)
    n = 1 << 14
    o = rng.uniform(-0.9, 0.9, (n, 3)) * np.array([1.0, 1.0, 0.1])
    d = rng.normal(size=(n, 3))
    rays = torch.as_tensor(np.concatenate([o, d / np.linalg.norm(d, axis=1, keepdims=True)], 1).astype(np.float32)).cuda()
    _, saved, _ = om.train_fwd(gpu_scene(sc, eps=0.12, n_max=2, t_thr=0.0), rays, torch.zeros(n, 3, device="cuda"))
    T = saved.view(-1, 20)[:8192, 7]
    T = T[(T > 1e-4) & (T < 0.3)].sort().values
    assert T.numel() > 1000
    for q in np.linspace(0, T.numel() - 1, 8).astype(int):
        t = np.float32(T[int(q)].item())
        for thr in (np.nextafter(t, np.float32(0)), t, np.nextafter(t, np.float32(1))):
            scene = gpu_scene(sc, eps=0.12, t_thr=float(thr))
            _, queue = om.render(scene, rays=rays)
            _, short = om.render(scene, rays=rays[:8192].contiguous())
            assert torch.equal(short, queue[:8192])


@pytest.mark.parametrize("w,h", [(1, 1), (1, 701), (2, 301), (3, 99), (4, 97), (701, 1), (301, 2), (99, 3), (2, 2), (6, 1),
                                 (5, 2)])
def test_narrow_images(w, h):
    """Images of a few columns or rows have super-tiles of their own: the same
    pixels in every form, and the counts of the 8 x 4 tiles in the queue (those
    that training saves), a good part of them decided by rounding."""
    scene = gpu_scene(_fog(0.004, holes=True), t_thr=0.3)
    cam = _camera(w, h)
    if w > 8 * h:
        cam["fx"] = cam["fy"] = np.float32(w)
    tiled, back = _tiles(oracle.camera_rays(cam), w, h)
    _, saved, _ = om.train_fwd(scene, tiled, torch.zeros(tiled.shape[0], 3, device="cuda"))
    want = saved.view(-1, 20)[:, 8].contiguous().view(torch.int32)[back]
    rgb, cnt = om.render(scene, camera=cam)
    assert torch.equal(cnt, want)
    assert torch.equal(om.render(scene, camera=cam, want_count=False)[0], rgb)
    for fill in (_camera(512, 300), _camera(1024, 1024)):
        g_rgb, g = om.render_cameras(scene, [cam, fill, cam])
        assert torch.equal(g[: w * h], want) and torch.equal(g_rgb[: w * h], rgb)
        assert torch.equal(g[-w * h:], want) and torch.equal(g_rgb[-w * h:], rgb)
        p_rgb, _ = om.render_cameras(scene, [cam, fill], want_count=False)
        assert torch.equal(p_rgb[: w * h], rgb)
    if w * h > 6:  # (fewer listed rays go through the queue)
        rays = torch.as_tensor(oracle.camera_rays(cam)).cuda()
        assert torch.equal(om.render(scene, rays=rays[:4096].contiguous(), want_count=False)[0], rgb[:4096])
