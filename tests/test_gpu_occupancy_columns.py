"""The occupancy grid where its columns are few, tall or in rows shorter than a
warp: the words against the oracle, and no shape left to a handful of warps."""
import numpy as np
import pytest
import torch

import oracle
import paper_2404_09531_gb300 as om

pytestmark = pytest.mark.gpu

AABB = (-1.0, 1.0, -1.0, 1.0, -0.125, 0.125)


@pytest.mark.parametrize("M", [1, 7, 40])
@pytest.mark.parametrize("N", [(1, 1, 1), (1, 1, 33333), (3, 5, 2049), (2, 33, 1000), (40, 3, 70), (1, 2, 22400),
                               (33, 31, 129), (150, 1, 31), (1, 150, 65)])
def test_few_tall_and_narrow_columns(N, M):
    rng = np.random.default_rng(11)
    occ = np.sort(rng.uniform(-0.15, 0.15, (M, M, 2)).astype(np.float32), axis=-1)
    edges = (np.float32(-0.125) + np.arange(N[2] + 1, dtype=np.float32) * np.float32(0.25 / N[2])).astype(np.float32)
    occ[::2] = np.sort(edges[rng.integers(0, N[2] + 1, occ[::2].shape)], axis=-1)
    occ[M // 2, M // 3] = (1.0, -1.0)
    bits, count = om.occupancy_grid(AABB, torch.as_tensor(occ).cuda(), N)
    ref, ref_count = oracle.occupancy_grid(AABB, occ, N)
    np.testing.assert_array_equal(om.unpack_occupancy_bits(bits, N[2]), ref.astype(bool))
    assert int(count.item()) == ref_count


def test_one_column_is_spread_over_the_chip():
    """2^24 voxels in one column take about as long as in 4,096 columns; one
    warp alone would take a hundred times as long."""
    occ = torch.tensor([[[-0.1, 0.1]]], device="cuda")

    def fastest(N):
        times = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            om.occupancy_grid(AABB, occ, N)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    assert fastest((1, 1, 1 << 24)) <= 5 * fastest((64, 64, 4096)) + 0.1


def test_the_tallest_column():
    """Voxel indices beyond 2^30, in one column: the count against the rule in
    torch's float32 (each operation rounded, as the definition has it)."""
    n = 2 ** 31 - 64
    z = (-0.1, 0.1)
    bits, count = om.occupancy_grid(AABB, torch.tensor([[z]], device="cuda"), (1, 1, n))
    hz = torch.tensor(0.25, device="cuda") / n
    z0 = torch.tensor(AABB[4], device="cuda")
    lo, hi = (torch.tensor(v, device="cuda") for v in z)
    want = 0
    for k0 in range(0, n, 1 << 27):
        k = torch.arange(k0, min(k0 + (1 << 27), n) + 1, device="cuda", dtype=torch.int64)
        e = z0 + k.float() * hz
        want += int(((lo < e[1:]) & (hi > e[:-1])).sum())
    assert int(count.item()) == want
