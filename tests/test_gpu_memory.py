"""Device memory that the faster paths take and the others do without: together at most an eighth of the
device's, and given back when a call on the object that holds it runs out of memory."""
import numpy as np
import pytest

import scangen
from tests.helpers import lib_grid

pytestmark = pytest.mark.gpu

RNG = np.random.default_rng(100)
SCAN = np.stack([RNG.uniform(-30, 30, 2000), RNG.uniform(-30, 30, 2000), RNG.uniform(-0.5, 5, 2000)], 1).astype(np.float32)
POSES = RNG.uniform(-1, 1, (10, 6)) * np.array([2, 2, 0.5, 0.05, 0.05, 0.2])


def _large(feature=1, **kw):
    """6.25M voxels: ten scattered poses hold 1.0 GB of sums."""
    from paper_1709_06948_gb300 import align
    spec = scangen.GridSpec(origin=(-40.0, -39.0625, -1.0), res_m=0.2, dims=(400, 390, 40), feature=feature, **kw)
    L = lib_grid(spec)
    align.align_set_reference(L, SCAN)
    return L


def test_grids_together_hold_a_share():
    import torch
    from paper_1709_06948_gb300 import align
    share = torch.cuda.get_device_properties(0).total_memory // 8
    sums = 10 * 400 * 390 * 40 * 16
    grids, kinds, results = [], [], set()
    for _ in range(share // sums + 2):
        L = _large(var_levels=1)
        mi, am, _ = align.align_eval_mi(L, SCAN, eta6=POSES)
        grids.append(L)
        kinds.append(align.align_eval_stats(L)["sweep"])
        results.add((mi.tobytes(), am))
    n = kinds.index(0)
    assert share // sums - 4 <= n <= share // sums and kinds == [4] * n + [0] * (len(kinds) - n)
    assert len(results) == 1
    # what a destroyed grid held can be taken again; a grid that holds its own keeps it
    grids[0].close()
    for L, kind in ((grids[-1], 4), (grids[-2], kinds[-2]), (grids[1], 4)):
        mi, am, _ = align.align_eval_mi(L, SCAN, eta6=POSES)
        assert align.align_eval_stats(L)["sweep"] == kind and (mi.tobytes(), am) in results
    for L in grids[1:]:
        L.close()


def test_given_back_when_memory_runs_out():
    """A grid that holds 1 GB of sums, a call that needs 0.66 GB of histograms, 0.3 GB free: the call
    succeeds, as it does with memory to spare, and the next scattered call takes its sums again."""
    import torch
    from paper_1709_06948_gb300 import align
    L = _large(feature=2, count_levels=7, var_levels=9)  # 64 symbols: 16 KB of histogram per pose
    many = np.random.default_rng(101).uniform(-1, 1, (40000, 6)) * np.array([2, 2, 0.5, 0.05, 0.05, 0.2])
    few = align.align_eval_mi(L, SCAN, eta6=POSES)
    assert align.align_eval_stats(L)["sweep"] == 4
    align.align_eval_mi(L, SCAN, eta6=many[:100])  # the table kernels' own buffers
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (300 << 20), dtype=torch.uint8, device="cuda")
    try:
        got = align.align_eval_mi(L, SCAN, eta6=many)
    finally:
        del fill
        torch.cuda.empty_cache()
    want = align.align_eval_mi(L, SCAN, eta6=many)
    assert np.array_equal(got[0].view(np.int32), want[0].view(np.int32)) and got[1] == want[1]
    again = align.align_eval_mi(L, SCAN, eta6=POSES)
    assert align.align_eval_stats(L)["sweep"] == 4 and np.array_equal(few[0].view(np.int32), again[0].view(np.int32))
    L.close()


def test_batch_gives_back_when_memory_runs_out():
    """The same for a batch's lattice workspace (70 MB; 689 MB of histograms, of which 35 are held, into 625
    free), and its graph afterwards."""
    import torch
    from paper_1709_06948_gb300 import align
    pair = scangen.lidar_pair(seed=scangen.SEED_BASE + 102, n_beams=32)
    spec = scangen.GridSpec(origin=(-40.0, -40.0, -1.0), res_m=0.25, dims=(320, 320, 32), feature=2, count_levels=7, var_levels=9)
    L = lib_grid(spec)
    align.align_set_reference(L, pair.xyzA)
    axes = [np.linspace(-h, h, m) for h, m in zip((2, 2, 0.2, 0.01, 0.01, 0.08), (8, 8, 2, 2, 2, 4))]
    lat = np.stack(np.meshgrid(*axes, indexing="ij"), -1).reshape(-1, 6)
    many = np.random.default_rng(103).uniform(-1, 1, (40000, 6)) * np.array([2, 2, 0.5, 0.05, 0.05, 0.2])
    b = align.align_batch_create()
    small, large = [(L, pair.xyzB, lat), (L, pair.xyzB[:100], many[:100])], [(L, pair.xyzB, lat), (L, pair.xyzB[:100], many)]
    first = align.align_eval_batch(b, small, graph=True)
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (625 << 20), dtype=torch.uint8, device="cuda")
    try:
        got = align.align_eval_batch(b, large, graph=True)
    finally:
        del fill
        torch.cuda.empty_cache()
    for pairs, res in ((large, got), (small, first)):
        for (mi, am), (mi0, am0) in zip(align.align_eval_batch(b, pairs, graph=True), res):
            assert np.array_equal(mi.view(np.int32), mi0.view(np.int32)) and am == am0
    align.align_batch_destroy(b)
    L.close()
