"""Kernels at the sizes where their dispatch or their tiling changes."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2404_09531_gb300 as om
from _util import brick_inputs, gpu_scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(1,), (3, 4, 5), (7, 1024, 883), (4097, 2, 64)])
@pytest.mark.parametrize("shift", [0, 1])
def test_adam_ragged_and_unaligned_groups(sizes, shift):
    """Groups of any size, and arrays 4 bytes off a 16-byte boundary (scalar
    accesses): the same bits as 4-byte steps in torch's float32."""
    gen = torch.Generator(device="cuda").manual_seed(7)
    groups, before = [], []
    for i, n in enumerate(sizes):
        g = {k: torch.randn(n + 4, device="cuda", generator=gen)[shift:shift + n] for k in ("param", "grad", "m", "v")}
        g["v"].abs_()
        g["lr"] = 1e-2
        if i % 2 == 0:
            g["shadow"] = torch.zeros(n + 4, dtype=torch.bfloat16, device="cuda")[shift:shift + n]
        groups.append(g)
        before.append({k: g[k].double().cpu().numpy() for k in ("param", "grad", "m", "v")})
    om.adam_step(groups, step=3, eps=1e-8)
    for g, b in zip(groups, before):
        m = 0.9 * b["m"] + 0.1 * b["grad"]
        v = 0.99 * b["v"] + 0.01 * b["grad"] ** 2
        p = b["param"] - 1e-2 / (1 - 0.9 ** 3) * m / (np.sqrt(v / (1 - 0.99 ** 3)) + 1e-8)
        # beta and its complement are rounded to float32 (2^-24 each), as are the
        # products and the sums; |m|, |v|, |p| are below 25
        for k, ref in (("m", m), ("v", v), ("param", p)):
            assert np.abs(g[k].cpu().numpy() - ref).max() <= 25 * 8 * 2.0 ** -24
        if "shadow" in g:
            assert torch.equal(g["shadow"], g["param"].to(torch.bfloat16))


@pytest.mark.parametrize("L", [(16, 16, 16), (257, 255, 31), (513, 520, 33)])
def test_brick_scan_over_several_rounds(L):
    """Tables below and above the 16,384 flags of one scan round."""
    spec = synth.scene_spec(2, L=L)
    occ = synth.make_scene(synth.scene_spec(2, L=(16, 16, 16), R=(16, 16, 16)))["occ"]
    table, n = om.build_brick_table(spec.aabb, L, 8, torch.as_tensor(occ).cuda())
    ref = oracle.brick_table(spec, occ)
    np.testing.assert_array_equal(table.cpu().numpy(), ref)
    assert int(n.item()) == ref.max() + 1


@pytest.mark.parametrize("N", [(33, 31, 1), (64, 32, 65), (90, 100, 129), (600000, 1, 3)])
def test_occupancy_grid_columns(N):
    """Columns in one cell and in several, ragged rows of 32, several words;
    the last size needs 64-bit cell arithmetic (M = 4096).  The intervals
    include voxel edges themselves, empty cells and infinities."""
    M = 4096 if N[0] > 1000 else 32
    rng = np.random.default_rng(3)
    occ = np.sort(rng.uniform(-0.2, 0.2, (M, M, 2)).astype(np.float32), axis=-1)
    edges = (np.float32(-0.125) + np.arange(N[2] + 1, dtype=np.float32) * np.float32(0.25 / N[2])).astype(np.float32)
    k = rng.integers(0, N[2] + 1, (M, M // 2, 2))
    occ[:, ::2] = np.sort(edges[k], axis=-1)
    occ[0, 0], occ[1, 1], occ[2, 2] = (1.0, -1.0), (-np.inf, np.inf), (0.0, 0.0)
    aabb = (-1.0, 1.0, -1.0, 1.0, -0.125, 0.125)
    bits, count = om.occupancy_grid(aabb, torch.as_tensor(occ).cuda(), N)
    ref, ref_count = oracle.occupancy_grid(aabb, occ, N)
    np.testing.assert_array_equal(om.unpack_occupancy_bits(bits, N[2]), ref.astype(bool))
    assert int(count.item()) == ref_count


@pytest.mark.parametrize("cfg", [3, 2])
@pytest.mark.parametrize("n", [1, 15, 17, 129, 4099])
def test_small_training_batches(cfg, n):
    """Batches that give a warp 4 to 32 rays: loss and gradients against the
    oracle's at the training tests' bar (1e-3 of the tensor's norm and largest
    value)."""
    sc = synth.make_scene(cfg)
    table, pool = brick_inputs(sc) if sc["spec"].brick else (None, None)
    if pool is not None:
        sc = dict(sc, grid=pool, table=table)
    scene = gpu_scene(sc)
    batch = synth.make_train_batch(cfg, n, K=2)
    lam = (1.0, 1e-2, 1e-4)
    res = om.train_step(scene, batch["rays"], batch["target"], batch["smooth_dirs"], lam=lam)
    ref = oracle.train(oracle.OracleScene(sc), batch["rays"], batch["target"], batch["smooth_dirs"], lam=lam)
    assert abs(float(res["loss"][0]) - ref["loss"]) <= 1e-5 * abs(ref["loss"])
    for k, g in res["grads"].items():
        a, b = g.double().cpu().numpy().ravel(), np.asarray(ref["grads"][k], np.float64).ravel()
        assert np.linalg.norm(a - b) <= 1e-3 * np.linalg.norm(b), k
        assert np.abs(a - b).max() <= 1e-3 * np.abs(b).max(), k


def test_gradient_of_a_bad_ray_stays_in_its_texels():
    """A ray with a NaN target makes its own texels' gradients NaN and leaves
    every other ray's texels as they are without it."""
    sc = synth.make_scene(3)
    scene = gpu_scene(sc)
    batch = synth.make_train_batch(3, 64, K=0)
    rays, target = batch["rays"], batch["target"].copy()
    good = om.train_step(scene, rays, target, None, lam=(1.0, 0.0, 0.0))["grads"]
    only = om.train_step(scene, rays[20:21], target[20:21], None, lam=(1.0, 0.0, 0.0))["grads"]
    target[20] = np.nan
    bad = om.train_step(scene, rays, target, None, lam=(1.0, 0.0, 0.0))["grads"]
    for k in ("grid", "p_xy", "p_xz", "p_yz"):
        away = only[k] == 0  # texels that ray does not reach
        assert torch.isfinite(bad[k][away]).all()
        # atomic additions in another order: a few roundings of the largest value
        assert (bad[k][away] - good[k][away]).abs().max() <= 64 * 2.0 ** -24 * good[k].abs().max()
    assert torch.isnan(bad["p_xy"]).any()
