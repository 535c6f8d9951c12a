"""Precision of the FP32 render's parts, against 64-bit values: no form of the
render may be coarser than float32 arithmetic in the plain order."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2404_09531_gb300 as om
from _util import gpu_scene

pytestmark = pytest.mark.gpu


def _camera(width, height, base=0):
    cam = synth.make_cameras(1)[base]
    f = np.float32(float(cam["fy"]) * height / float(cam["height"]))
    return dict(cam, width=width, height=height, fx=f, fy=f, cx=np.float32(0.5 * width), cy=np.float32(0.5 * height))


def _colourless_scene(mlp):
    """Opaque everywhere, diffuse colour and features 0: a pixel is the MLP's output."""
    sc = synth.make_scene(1)
    for k in ("grid", "p_xy", "p_xz", "p_yz"):
        sc[k] = np.zeros_like(sc[k])
    sc["grid"][..., 0] = 8.0
    sc["grid"][..., 1:] = -80.0
    sc["occ"] = np.full_like(sc["occ"], 10.0) * np.array([-1.0, 1.0], np.float32)
    sc["mlp"] = mlp
    return gpu_scene(sc)


@pytest.mark.parametrize("power", [0, 1, 2, 3])
@pytest.mark.parametrize("cosine", [0, 1])
def test_view_encoding(power, cosine):
    """Output c is sigmoid(256 f) of one value f = sin or cos of 2^power d_c, an
    exact product: the hidden units pass f and -f on, and relu(f) - relu(-f) = f.
    sincosf is within 2 ulp, which |256 f| sigmoid' makes at most 0.23 * 2^-22;
    the sigmoid's own operations (expf, sum, quotient: 4 ulp at most) 4 * 2^-24."""
    mlp = np.zeros(883, np.float32)
    W1, W2, W3 = mlp[:544].reshape(16, 34), mlp[560:816].reshape(16, 16), mlp[832:880].reshape(3, 16)
    W2[:] = np.eye(16)
    for c in range(3):
        W1[2 * c, 10 + 6 * power + 3 * cosine + c] = 1.0
        W1[2 * c + 1, 10 + 6 * power + 3 * cosine + c] = -1.0
        W3[c, 2 * c], W3[c, 2 * c + 1] = 256.0, -256.0
    scene = _colourless_scene(mlp)
    tol = 0.23 * 2.0 ** -22 + 4 * 2.0 ** -24

    def check(rgb, cnt, rays):
        d = np.asarray(rays, np.float32)[:, 3:].astype(np.float64) * 2.0 ** power
        f = np.cos(d) if cosine else np.sin(d)
        want = 1.0 / (1.0 + np.exp(-256.0 * f))
        hit = cnt.cpu().numpy() > 0
        assert hit.mean() > 0.2
        assert np.abs(rgb.cpu().numpy() - want)[hit].max() <= tol

    for n in (2000, 20000):  # 8 lanes per ray, the queue
        rng = np.random.default_rng(n)
        o = rng.uniform(-0.5, 0.5, (n, 3)) * np.array([1.0, 1.0, 0.1])
        d = rng.normal(0.0, 1.0, (n, 3))
        d *= rng.choice([1.0, 4.0], (n, 1)) / np.linalg.norm(d, axis=1, keepdims=True)
        rays = np.concatenate([o, d], 1).astype(np.float32)
        rgb, cnt = om.render(scene, rays=rays)
        check(rgb, cnt, rays)
    for w, h in ((97, 61), (512, 300), (1024, 801)):  # 8, 4 and 1 lanes per ray
        cam = _camera(w, h)
        rgb, cnt = om.render(scene, camera=cam)
        check(rgb, cnt, oracle.camera_rays(cam))


@pytest.mark.parametrize("sigma", [0.004, 0.012, 0.1])
def test_sums_over_long_rays(sigma):
    """Rays of many samples in fog of about the optical depth sigma per sample:
    the camera's forms and short lists are no coarser against the oracle than
    the packed queue, whose lane scans round each contribution a few times only
    (5 % for the spread of 6,000 rays' errors)."""
    spec = synth.scene_spec(1, step=1.0 / 4096, n_max=2048)
    sc = synth.make_scene(spec)
    density = np.log(sigma * 4096) + 0.1 * np.random.default_rng(3).normal(size=sc["grid"].shape[:3])
    sc["grid"][..., 0] = density.astype(np.float32)
    for k in ("p_xy", "p_xz", "p_yz"):
        sc[k][..., 0] = 0.0
    sc["occ"] = np.full_like(sc["occ"], 0.12) * np.array([-1.0, 1.0], np.float32)
    sc["mlp"] = np.zeros_like(sc["mlp"])
    scene = gpu_scene(sc)
    cam = _camera(96, 64)
    n = 96 * 64
    rays = torch.as_tensor(oracle.camera_rays(cam)).cuda()
    ref = oracle.render(oracle.OracleScene(sc), rays.cpu().numpy())
    ok = torch.as_tensor(ref["ambiguous"] == 0).cuda()
    want = torch.as_tensor(ref["rgb"]).cuda()

    def rms(rgb):
        return float((rgb[:n].double() - want)[ok].pow(2).mean().sqrt())

    queue = rms(om.render(scene, rays=torch.cat([rays] * 3), want_count=False)[0])
    assert rms(om.render(scene, camera=cam, want_count=False)[0]) <= 1.05 * queue
    assert rms(om.render(scene, rays=rays, want_count=False)[0]) <= 1.05 * queue
    for fill in (_camera(512, 300), _camera(1024, 801)):
        assert rms(om.render_cameras(scene, [cam, fill], want_count=False)[0]) <= 1.05 * queue
