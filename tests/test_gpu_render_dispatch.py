"""Renders on both sides of every line of the dispatch (lanes per ray by the rays
of the launch, the box's height in lattice steps and whether counts are wanted;
short lists): the same pixels and counts."""
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


def _scene(cfg):
    sc = synth.make_scene(cfg)
    table, pool = brick_inputs(sc) if sc["spec"].brick else (None, None)
    return sc, table, pool, gpu_scene(sc, table=table)


# (rays - 1 and rays) of the lines, without and with counts
LINES = {1: ((5 << 14, 5 << 16), (5 << 14, 3 << 16)), 2: ((1 << 17, 3 << 18), (1 << 17, 7 << 16))}


@pytest.mark.parametrize("cfg", [1, 2])
@pytest.mark.parametrize("count", [False, True])
def test_launches_beside_the_lines(cfg, count):
    _, _, _, scene = _scene(cfg)
    probe = _camera(cfg, 61, 41)
    n = 61 * 41
    want, want_cnt = om.render(scene, camera=probe)
    for line in LINES[cfg][count]:
        for total in (line - 1, line):
            rest = total - n
            fill = _camera(cfg, 256, rest // 256)
            last = _camera(cfg, rest % 256, 1) if rest % 256 else None
            rgb, cnt = om.render_cameras(scene, [probe, fill] + ([last] if last else []), want_count=count)
            assert rgb.shape[0] == total
            assert torch.equal(rgb[:n], want)
            if count:
                assert torch.equal(cnt[:n], want_cnt)


@pytest.mark.parametrize("cfg", [1, 2])
@pytest.mark.parametrize("n", [1, 5, 6, 7, 8])
def test_a_handful_of_listed_rays(cfg, n):
    sc, table, pool, scene = _scene(cfg)
    rays = synth.make_train_batch(cfg, 4096, K=1)["rays"]
    for at in (0, 1000, 2048):
        part = np.ascontiguousarray(rays[at:at + n])
        rgb, cnt = om.render(scene, rays=part)
        assert torch.equal(om.render(scene, rays=part, want_count=False)[0], rgb)
        ref = oracle.render(oracle_scene_for(sc, table, pool), part)
        if (ref["ambiguous"] == 0).all():
            compare_render(rgb.cpu().numpy(), cnt.cpu().numpy(), ref, what=f"config {cfg}, {n} rays")
