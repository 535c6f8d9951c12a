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
