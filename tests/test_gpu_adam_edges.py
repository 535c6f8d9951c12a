"""Adam over arrays on and off a 16-byte boundary: the right values and nothing
written beside them."""
import numpy as np
import pytest
import torch

import paper_2404_09531_gb300 as om

pytestmark = pytest.mark.gpu

PAD = 8  # elements kept free on both sides of every array


def _groups(sizes, shifts, seed=5):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    backing, groups = [], []
    for i, (n, shift) in enumerate(zip(sizes, shifts)):
        b = {k: torch.randn(n + 2 * PAD, device="cuda", generator=gen) for k in ("param", "grad", "m", "v")}
        b["v"].abs_()
        if i % 2 == 0:
            b["shadow"] = torch.randn(n + 2 * PAD, device="cuda", generator=gen).to(torch.bfloat16)
        backing.append((b, PAD + shift, n))
        groups.append(dict({k: t[PAD + shift:PAD + shift + n] for k, t in b.items()}, lr=1e-2))
    return backing, groups


@pytest.mark.parametrize("sizes,shifts", [((1, 2, 3), (0, 1, 2)), ((5, 7, 883), (0, 3, 1)), ((1030, 0, 257, 4099, 129, 130), (1, 0, 0, 2, 0, 3))])
def test_mixed_groups_and_their_neighbourhood(sizes, shifts):
    backing, groups = _groups(sizes, shifts)
    before = [{k: t.clone() for k, t in b.items()} for b, _, _ in backing]
    om.adam_step(groups, step=3, eps=1e-8)
    for (b, at, n), old in zip(backing, before):
        for k, t in b.items():
            keep = torch.ones(t.numel(), dtype=torch.bool, device="cuda")
            keep[at:at + n] = k == "grad"
            assert torch.equal(t[keep], old[k][keep]), k
        w = {k: old[k][at:at + n].double().cpu().numpy() for k in ("param", "grad", "m", "v")}
        m = 0.9 * w["m"] + 0.1 * w["grad"]
        v = 0.99 * w["v"] + 0.01 * w["grad"] ** 2
        p = w["param"] - 1e-2 / (1 - 0.9 ** 3) * m / (np.sqrt(v / (1 - 0.99 ** 3)) + 1e-8)
        # the rounded betas, products and sums: 8 roundings of values below 25
        for k, ref in (("m", m), ("v", v), ("param", p)):
            assert np.abs(b[k][at:at + n].cpu().numpy() - ref).max(initial=0.0) <= 25 * 8 * 2.0 ** -24, k
        if "shadow" in b:
            assert torch.equal(b["shadow"][at:at + n], b["param"][at:at + n].to(torch.bfloat16))
