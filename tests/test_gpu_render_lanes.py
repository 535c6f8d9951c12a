"""The camera render's forms (8, 4 or 1 lanes per ray, chosen by the number of
rays of a launch): a camera's pixels and counts are the same in every form,
with and without counts, and match the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2404_09531_gb300 as om
from _util import brick_inputs, compare_render, gpu_scene, oracle_scene_for

pytestmark = pytest.mark.gpu


def _camera(cfg, width, height):
    cam = synth.make_cameras(cfg)[0]
    f = np.float32(float(cam["fy"]) * height / float(cam["height"]))
    return dict(cam, width=width, height=height, fx=f, fy=f, cx=np.float32(0.5 * width), cy=np.float32(0.5 * height))


@pytest.mark.parametrize("cfg", [1, 2])
@pytest.mark.parametrize("size", [(1, 1), (37, 23), (64, 50), (131, 67)])
def test_every_form_gives_the_same_pixels(cfg, size):
    sc = synth.make_scene(cfg)
    table, pool = brick_inputs(sc) if sc["spec"].brick else (None, None)
    scene = gpu_scene(sc, table=table)
    cam = _camera(cfg, *size)
    n = size[0] * size[1]
    rgb, cnt = om.render(scene, camera=cam)  # fewer than 2^17 rays
    ref = oracle.render(oracle_scene_for(sc, table, pool), oracle.camera_rays(cam))
    compare_render(rgb.cpu().numpy(), cnt.cpu().numpy(), ref, what=f"config {cfg} {size}")
    # the same camera in launches of 2^17 and of 2^20 or more rays
    for fill in (_camera(cfg, 512, 256), _camera(cfg, 1024, 1024)):
        g_rgb, g_cnt = om.render_cameras(scene, [fill, cam])
        assert torch.equal(g_rgb[-n:], rgb) and torch.equal(g_cnt[-n:], cnt)
        p_rgb, _ = om.render_cameras(scene, [cam, fill], want_count=False)
        assert torch.equal(p_rgb[:n], rgb)
        assert torch.equal(p_rgb[n:], g_rgb[:-n])


@pytest.mark.parametrize("cfg", [1, 2])
@pytest.mark.parametrize("n", [1, 17, 1000, 16383])
def test_short_ray_lists_match_long_ones(cfg, n):
    """Fewer than 2^14 rays take 8 lanes each, more the packed queue: the same
    counts, and pixels within the rounding of the two orders of summation."""
    sc = synth.make_scene(cfg)
    table, pool = brick_inputs(sc) if sc["spec"].brick else (None, None)
    scene = gpu_scene(sc, table=table)
    rays = torch.as_tensor(synth.make_train_batch(cfg, 16384, K=1)["rays"]).cuda()
    long_rgb, long_cnt = om.render(scene, rays=rays)
    rgb, cnt = om.render(scene, rays=rays[:n].contiguous())
    only_rgb, _ = om.render(scene, rays=rays[:n].contiguous(), want_count=False)
    assert torch.equal(cnt, long_cnt[:n])
    assert torch.equal(only_rgb, rgb)
    # about 50 sums of values below 1, each rounded by 2^-24, in either order
    assert (rgb - long_rgb[:n]).abs().max().item() <= 2 * 50 * 2.0 ** -24
    idx = np.arange(0, n, max(1, n // 500))
    r = rays[:n].cpu().numpy()[idx]
    ref = oracle.render(oracle_scene_for(sc, table, pool), r)
    compare_render(rgb.cpu().numpy()[idx], cnt.cpu().numpy()[idx], ref, what=f"config {cfg}, {n} rays")


def test_counts_where_rounding_decides_the_termination():
    """A constant density makes every ray's transmittance after 20 samples the
    same but for rounding, and the termination threshold is its median: the
    order of the products decides the counts.  Cameras in every form and short
    ray lists give the counts of the packed queue, which marches the same 8 x 4
    tiles as a list of 2^14 rays."""
    sc = synth.make_scene(1)
    for k in ("grid", "p_xy", "p_xz", "p_yz"):
        sc[k] = np.zeros_like(sc[k])
    sc["grid"][..., 0] = 3.0
    sc["occ"] = np.full_like(sc["occ"], 10.0) * np.array([-1.0, 1.0], np.float32)  # no ramp inside the box
    w, h = 256, 64
    cam = _camera(1, w, h)
    rays = oracle.camera_rays(cam).reshape(h // 4, 4, w // 8, 8, 6).transpose(0, 2, 1, 3, 4).reshape(-1, 6)
    rays = torch.as_tensor(np.ascontiguousarray(rays)).cuda()
    # the queue's transmittances after exactly 20 samples (the saved training state)
    _, saved, _ = om.train_fwd(gpu_scene(sc, t_thr=0.0, n_max=20), rays, torch.zeros(rays.shape[0], 3, device="cuda"))
    state = saved.view(-1, 20)
    after = state[state[:, 8].contiguous().view(torch.int32) == 20, 7]
    scene = gpu_scene(sc, t_thr=float(after.median()))
    rgb, cnt = om.render(scene, camera=cam)
    _, queue = om.render(scene, rays=rays)  # 2^14 rays, 32 to a tile
    tiled = queue.view(h // 4, w // 8, 4, 8).permute(0, 2, 1, 3).reshape(-1)
    # the threshold does split the rays by rounding
    assert (queue == 20).sum() >= 20 and (queue == 21).sum() >= 20
    assert torch.equal(cnt, tiled)
    for fill in (_camera(1, 512, 256), _camera(1, 1024, 1024)):
        _, g = om.render_cameras(scene, [fill, cam])
        assert torch.equal(g[-w * h:], tiled)
    for n in (1, 40, 5000):
        _, short = om.render(scene, rays=rays[:n].contiguous())
        assert torch.equal(short, queue[:n])
