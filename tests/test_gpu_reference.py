"""A's prefix sums from the list of its occupied voxels: the marginals of A over any overlap box, at the
edges of the strips and warps they are written in."""
import numpy as np
import pytest

import oracle
import scangen
from tests.helpers import lib_grid, mi_tolerance, oracle_grid

pytestmark = pytest.mark.gpu


# with 56 symbols (feature 2) all but the first two and the widest take the list
@pytest.mark.parametrize("dims,res", [((1, 1, 1), 4.0), ((33, 65, 7), 0.7), ((31, 63, 80), 0.3), ((32, 64, 80), 0.3),
                                      ((33, 61, 90), 0.3), ((160, 66, 16), 0.1), ((161, 62, 17), 0.1),
                                      ((416, 130, 3), 0.1), ((417, 130, 3), 0.1), ((2048, 9, 8), 0.02),
                                      ((2049, 9, 8), 0.02), ((5, 300, 90), 0.2)])
@pytest.mark.parametrize("feature", [0, 1, 2])
def test_reference_symbols_and_marginals(dims, res, feature):
    """Histograms (their phi column and A's row sums come from the prefix sums) against the oracle, for
    two references in turn on one grid (the second finds the sums cleared) and an empty one."""
    from paper_1709_06948_gb300 import align
    rng = np.random.default_rng(sum(dims) + feature)
    size = np.array(dims) * res
    spec = scangen.GridSpec(origin=tuple(-size / 2), res_m=res, dims=dims, feature=feature, count_levels=7,
                            var_levels=8 if feature == 2 else 15)
    L, G = lib_grid(spec), oracle_grid(spec)
    etas = rng.uniform(-0.3, 0.3, (12, 6)) * np.concatenate([size, np.full(3, 0.2)])
    poses = align.align_round_poses(spec.origin, etas)
    B = (rng.uniform(-0.5, 0.5, (3000, 3)) * size).astype(np.float32)
    for n in (4000, 700, 0):
        A = (rng.uniform(-0.55, 0.55, (n, 3)) ** 3 * 4 * size).astype(np.float32)
        align.align_set_reference(L, A)
        symA, boxA = G.reference(A)
        sym, box = align.align_get_reference(L)
        assert np.array_equal(sym, symA) and np.array_equal(box, boxA)
        mi, _, hist = align.align_eval_mi(L, B, eta6=etas, with_hist=True)
        mo, ho, _ = G.eval_mi(symA, boxA, B, poses, nthreads=oracle.host_cores(), with_hist=True)
        assert np.array_equal(hist, ho) and np.max(np.abs(mi.astype(np.float64) - mo)) <= mi_tolerance()
    L.close()


@pytest.mark.parametrize("dims,res", [((161, 62, 17), 0.1), ((160, 64, 17), 0.1), ((419, 131, 3), 0.1)])
@pytest.mark.parametrize("mixed", [True, False])
def test_reference_with_every_voxel_occupied(dims, res, mixed):
    """Sixteen symbols of a list thread's words all set, and the last thread's part of them (the sizes of
    the grids leave 14, 0 and 11 voxels for it): by list while no symbol has too many voxels (mixed counts
    and heights), by the passes when one has (one to three points per voxel)."""
    from paper_1709_06948_gb300 import align
    rng = np.random.default_rng(95)
    size = np.array(dims) * res
    spec = scangen.GridSpec(origin=tuple(-size / 2), res_m=res, dims=dims, feature=2, count_levels=7, var_levels=8)
    k = np.stack(np.meshgrid(*(np.arange(d) for d in dims), indexing="ij"), -1).reshape(-1, 3)
    n = 2 ** rng.integers(2, 7, len(k)) if mixed else rng.integers(1, 4, len(k))
    half = np.repeat(0.45 * 0.5 ** rng.uniform(0, 2.5, len(k)) if mixed else np.full(len(k), 0.2), n)
    k = np.repeat(k, n, axis=0)
    A = ((k + 0.5 + rng.uniform(-1, 1, k.shape) * half[:, None]) * res - size / 2).astype(np.float32)
    L, G = lib_grid(spec), oracle_grid(spec)
    align.align_set_reference(L, A)
    launches = align.align_eval_stats(L)["kernel_launches"]
    assert launches == (5 if mixed else 8)  # sums, symbols, and the list's three kernels (then the passes)
    symA, boxA = G.reference(A)
    assert np.count_nonzero(symA) == len(symA.reshape(-1))
    sym, box = align.align_get_reference(L)
    assert np.array_equal(sym, symA) and np.array_equal(box, boxA)
    etas = rng.uniform(-0.3, 0.3, (6, 6)) * np.concatenate([size, np.full(3, 0.1)])
    B = A[rng.integers(0, len(A), 4000)]
    _, _, hist = align.align_eval_mi(L, B, eta6=etas, with_hist=True)
    _, ho, _ = G.eval_mi(symA, boxA, B, align.align_round_poses(spec.origin, etas), nthreads=oracle.host_cores(),
                         with_hist=True)
    assert np.array_equal(hist, ho)
    L.close()
