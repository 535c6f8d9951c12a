"""Training batches in every band of the backward's dispatch: the re-march takes 4,
8, 16 or 32 rays per warp and a work counter once the warps' slots are full, the
MLP backward one or two tiles of 16 rays."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2404_09531_gb300 as om
from _util import GRAD_RTOL, gpu_scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def scene_and_batch():
    sc = synth.make_scene(3)
    return sc, gpu_scene(sc), synth.make_train_batch(3, 131072, K=1)


# Ragged batches, in rays per SM of the re-march's 20 warps each: 4 rays per warp
# below 160 rays per SM (a counter above 80), 8 below 320, 16 below 640 (above
# about 512 with two MLP tiles), 32 from there on
@pytest.mark.parametrize("per_sm", [100, 200, 400, 530, 700])
def test_ragged_batches(scene_and_batch, per_sm):
    sc, scene, batch = scene_and_batch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = min(per_sm * sms | 3, 131072 - 1)
    rays, target, dirs = batch["rays"][:n], batch["target"][:n], batch["smooth_dirs"][:n]
    lam = (1.0, 1e-2, 1e-4)
    res = om.train_step(scene, rays, target, dirs, lam=lam)
    ref = oracle.train(oracle.OracleScene(sc), rays, target, dirs, lam=lam)
    assert abs(float(res["loss"][0]) - ref["loss"]) <= 1e-5 * abs(ref["loss"])
    for k, g in res["grads"].items():
        a, b = g.double().cpu().numpy().ravel(), np.asarray(ref["grads"][k], np.float64).ravel()
        assert np.linalg.norm(a - b) <= GRAD_RTOL * np.linalg.norm(b), k
        assert np.abs(a - b).max() <= GRAD_RTOL * np.abs(b).max(), k
