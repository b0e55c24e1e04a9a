"""Poses that share nothing, their points spread over the GPU, against one pose per CTA and the oracle:
the same histograms and MI, at the edges of warps, blocks and of the 32-bit sums."""
import numpy as np
import pytest

import oracle
import scangen
from tests.helpers import check_argmax, lib_grid, mi_tolerance, oracle_grid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tiny():
    return scangen.tiny_pair()


def _check(spec, A, B, etas, sweep=4, **over):
    from paper_1709_06948_gb300 import align
    L = lib_grid(spec, **over)
    align.align_set_reference(L, A)
    for _ in range(2):  # the second call finds the sums cleared by the first
        mi, am, hist = align.align_eval_mi(L, B, eta6=etas, with_hist=True)
        st = align.align_eval_stats(L)
        assert st["sweep"] == sweep, st
        assert len(align.align_eval_redo_poses(L)) == 0 or sweep != 4
    align.align_set_sweep(L, 0)
    mi0, am0, hist0 = align.align_eval_mi(L, B, eta6=etas, with_hist=True)
    assert np.array_equal(mi.view(np.int32), mi0.view(np.int32)) and am == am0 and np.array_equal(hist, hist0)
    G = oracle_grid(spec, **over)
    symA, boxA = G.reference(A)
    poses = align.align_round_poses(spec.origin, etas)
    mo, ho, _ = G.eval_mi(symA, boxA, B, poses, nthreads=oracle.host_cores(), with_hist=True)
    assert np.array_equal(hist, ho) and np.max(np.abs(mi.astype(np.float64) - mo)) <= mi_tolerance()
    check_argmax(am, mo, mi)
    L.close()
    return st


def _poses(n, seed, scale=1.0):
    rng = np.random.default_rng(seed)
    return rng.uniform(-1, 1, (n, 6)) * np.array([2, 2, 0.5, 0.1, 0.1, 0.4]) * scale


@pytest.mark.parametrize("feature", [0, 1, 2])
@pytest.mark.parametrize("n_poses", [1, 2, 31, 32])
def test_few_poses(tiny, feature, n_poses):
    spec = scangen.GridSpec(origin=(-20.0, -20.0, -1.0), res_m=0.5, dims=(79, 83, 15), feature=feature,
                            count_levels=7, var_levels=8 if feature == 2 else 15)
    _check(spec, tiny.xyzA, tiny.xyzB, _poses(n_poses, 7 * n_poses + feature, 1.0 if n_poses < 31 else 12.0))


@pytest.mark.parametrize("n", [0, 1, 31, 33, 511, 513, 1025])
def test_point_counts_around_warps_and_blocks(tiny, n):
    _check(tiny.grid, tiny.xyzA, tiny.xyzB[:n], _poses(5, n))


def test_more_poses_keep_one_per_cta(tiny):
    _check(tiny.grid, tiny.xyzA, tiny.xyzB, _poses(33, 3), sweep=0)


@pytest.mark.parametrize("n_poses,sweep", [(16, 4), (17, 0)])
@pytest.mark.parametrize("feature", [0, 1])
def test_many_poses_on_few_voxels_keep_one_per_cta(tiny, n_poses, sweep, feature):
    spec = scangen.GridSpec(origin=(-20.0, -20.0, -1.0), res_m=8.0, dims=(5, 5, 2), feature=feature, count_levels=7)
    _check(spec, tiny.xyzA, tiny.xyzB, _poses(n_poses, 19), sweep=sweep)


def test_non_finite_points(tiny):
    xyz = tiny.xyzB.copy()
    xyz[::7, 0] = np.nan
    xyz[1::11, 1] = np.inf
    xyz[2::13, 2] = -np.inf
    _check(tiny.grid, tiny.xyzA, xyz, _poses(6, 5))


def test_dense_voxel_past_32_bit_sums():
    """70,000 points in one 0.5 m voxel: exact in the 64-bit sums, counted as wide."""
    rng = np.random.default_rng(93)
    spec = scangen.lidar_grid(0.5)
    xyz = np.concatenate([np.stack([rng.uniform(a, a + 0.2, 70000) for a in (1.15, 2.15, 0.15)], 1),
                          np.stack([rng.uniform(-30, 30, 3000), rng.uniform(-30, 30, 3000), rng.uniform(-0.5, 5, 3000)], 1)])
    xyz = xyz.astype(np.float32)
    st = _check(spec, xyz, xyz, _poses(3, 11, 0.02))
    assert st["wide_voxels"] >= 1


def test_calls_in_turn_leave_nothing_behind():
    """Table kernels with exact-path poses, then scattered calls of other sizes, places and outputs on the
    same grid: each as on a fresh one, and no pose of an earlier call listed as redone."""
    from paper_1709_06948_gb300 import align
    rng = np.random.default_rng(94)
    spec = scangen.lidar_grid(0.5)
    xyz = np.stack([rng.uniform(a, a + 0.2, 70000) for a in (1.15, 2.15, 0.15)], 1).astype(np.float32)
    L = lib_grid(spec)
    align.align_set_reference(L, xyz)
    align.align_set_sweep(L, 0)
    align.align_eval_mi(L, xyz, eta6=_poses(40, 12, 0.02))
    assert len(align.align_eval_redo_poses(L)) > 0
    align.align_set_sweep(L, -1)
    away = _poses(2, 17)
    away[:, 0] = 1000.0, -1000.0  # no point in the grid: an empty overlap
    for n, etas in ((70000, _poses(4, 13, 0.02)), (70000, away), (0, _poses(1, 14)), (9, _poses(9, 15)), (70000, _poses(2, 16))):
        got = align.align_eval_mi(L, xyz[:n], eta6=etas, with_hist=n != 9)
        assert align.align_eval_stats(L)["sweep"] == 4 and len(align.align_eval_redo_poses(L)) == 0
        F = lib_grid(spec)
        align.align_set_reference(F, xyz)
        align.align_set_sweep(F, 0)
        want = align.align_eval_mi(F, xyz[:n], eta6=etas, with_hist=n != 9)
        assert np.array_equal(got[0].view(np.int32), want[0].view(np.int32)) and got[1] == want[1]
        assert n == 9 or np.array_equal(got[2], want[2])
        F.close()
    L.close()
