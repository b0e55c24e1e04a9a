"""Pose lattices evaluated by groups (every combination of some rotations and t'_x, t'_y, t'_z) against
the table kernels and the oracle: the same MI bit for bit, at the edges of the groups, masks, chunks and
rounds that the path cuts its work into."""
import math

import numpy as np
import pytest

import oracle
import scangen
from tests.helpers import lib_grid, mi_tolerance, oracle_grid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tiny():
    return scangen.tiny_pair()


def _lattice(counts, half, order=(3, 4, 5, 0, 1, 2), centre=np.zeros(6)):
    axes = [np.array([c]) if m < 2 else c + np.linspace(-h, h, m) for c, h, m in zip(centre, half, counts)]
    g = np.meshgrid(*(axes[a] for a in order), indexing="ij")
    etas = np.empty((g[0].size, 6))
    for a, v in zip(order, g):
        etas[:, a] = v.reshape(-1)
    return etas


def _check(spec, A, B, etas, sweep=3, sample=24, **over):
    """MI and argmax by groups equal one pose per CTA's, and a sample the oracle's."""
    from paper_1709_06948_gb300 import align
    L = lib_grid(spec, **over)
    align.align_set_reference(L, A)
    mi, am, _ = align.align_eval_mi(L, B, eta6=etas)
    st = align.align_eval_stats(L)
    assert st["sweep"] == sweep, st
    redo = align.align_eval_redo_poses(L)
    align.align_set_sweep(L, 0)
    mi0, am0, _ = align.align_eval_mi(L, B, eta6=etas)
    assert np.array_equal(mi.view(np.int32), mi0.view(np.int32)) and am == am0
    pick = np.unique(np.concatenate([[am], np.linspace(0, len(etas) - 1, sample).astype(int)]))
    G = oracle_grid(spec, **over)
    symA, boxA = G.reference(A)
    mo, _, _ = G.eval_mi(symA, boxA, B, align.align_round_poses(spec.origin, etas[pick]), nthreads=oracle.host_cores())
    assert np.max(np.abs(mi[pick].astype(np.float64) - mo)) <= mi_tolerance()
    L.close()
    return redo


SMALL = (0.8, 0.7, 0.3, 0.02, 0.02, 0.05)


@pytest.mark.parametrize("counts,half,order", [
    ((2, 8, 2, 2, 2, 3), SMALL, (3, 4, 5, 0, 1, 2)),              # the fewest t'_x of a group
    ((3, 3, 3, 3, 3, 3), SMALL, (0, 1, 2, 3, 4, 5)),              # rotations fastest
    ((8, 20, 1, 2, 2, 2), (3.0, 2.0, 0.0, 0.01, 0.02, 0.03), (2, 1, 0, 3, 4, 5)),
    ((9, 13, 2, 2, 1, 3), SMALL, (5, 2, 0, 1, 3, 4)),             # two chunks of t'_x, 5 and 4
    ((17, 40, 2, 1, 1, 2), (9.0, 0.4, 0.1, 0.0, 0.0, 0.1), (3, 4, 5, 0, 1, 2)),
    ((70, 5, 1, 1, 1, 5), (30.0, 0.4, 0.0, 0.0, 0.0, 0.1), (3, 4, 5, 0, 1, 2)),  # two rounds of t'_x
    ((8, 8, 3, 1, 1, 8), (1e-4, 1e-4, 1e-3, 0.0, 0.0, 0.1), (3, 4, 5, 0, 1, 2)),  # nearly equal poses
    ((8, 8, 1, 2, 2, 5), (60.0, 60.0, 0.0, 0.5, 0.5, 3.0), (3, 4, 5, 0, 1, 2)),  # most poses leave the grid
])
@pytest.mark.parametrize("feature", [0, 1, 2])
def test_groups_equal_table_kernels(tiny, counts, half, order, feature):
    spec = scangen.GridSpec(origin=(-20.0, -20.0, -1.0), res_m=0.5, dims=(79, 83, 15), feature=feature,
                            count_levels=7, var_levels=8 if feature == 2 else 15)
    _check(spec, tiny.xyzA, tiny.xyzB, _lattice(counts, half, order, tiny.T))


@pytest.mark.parametrize("n", [0, 1, 31, 33, 255, 257, 4097])
def test_point_counts_around_warps_and_blocks(tiny, n):
    _check(tiny.grid, tiny.xyzA, tiny.xyzB[:n], _lattice((4, 20, 2, 1, 1, 4), SMALL))


@pytest.mark.parametrize("dims,res", [((1, 400, 3), 0.3), ((400, 1, 40), 0.2), ((33, 35, 64), 0.25), ((700, 90, 4), 0.1)])
def test_grid_shapes(tiny, dims, res):
    """One voxel column, one row, tall, and wide enough for groups of four t'_x."""
    spec = scangen.GridSpec(origin=(-dims[0] * res / 2, -dims[1] * res / 2, -1.0), res_m=res, dims=dims, feature=1,
                            var_levels=15)
    _check(spec, tiny.xyzA, tiny.xyzB, _lattice((8, 20, 2, 1, 1, 4), SMALL))


@pytest.mark.parametrize("feature,n", [(0, 8000), (1, 4000), (2, 8000), (2, 4000)])
def test_sparse_rows(tiny, feature, n):
    """Few points per row and tables that leave one CTA per SM: mask words only where there are cells."""
    spec = scangen.GridSpec(origin=(-25.0, -25.0, -1.0), res_m=0.1, dims=(500, 40, 10), feature=feature, count_levels=7,
                            var_levels=8 if feature == 2 else 15)
    squeeze = np.array([1.0, 0.1, 0.2], np.float32)  # a street 4 m wide
    _check(spec, tiny.xyzA * squeeze, np.ascontiguousarray(tiny.xyzB[:: 8000 // n] * squeeze), _lattice((7, 20, 2, 1, 1, 4), SMALL))


@pytest.mark.parametrize("feature", [0, 1, 2])
def test_rows_planned_again(feature):
    """Layers of points that share a few cells (chunks are planned ever larger) between layers of points
    with cells of their own: the chunk after each change holds more cells than planned and is planned
    again, with other rows' ends copied into the same words."""
    rng = np.random.default_rng(96)
    spec = scangen.GridSpec(origin=(-25.0, -3.0, 0.0), res_m=0.25, dims=(200, 24, 8), feature=feature, count_levels=7,
                            var_levels=8 if feature == 2 else 15)
    n = 24 * 600
    layers = []
    for k in range(8):
        x = rng.uniform(-24, 24, 10)[rng.integers(0, 10, n)] if k % 2 == 0 else rng.uniform(-24, 24, n)
        y = -2.875 + 0.25 * rng.integers(0, 24, n) if k % 2 == 0 else rng.uniform(-3, 3, n)
        layers.append(np.stack([x, y, np.full(n, 0.25 * k + 0.12) + rng.uniform(-0.1, 0.1, n) * (k % 2)], 1))
    xyz = np.concatenate(layers).astype(np.float32)
    _check(spec, xyz, xyz, _lattice((8, 20, 2, 1, 1, 4), (0.8, 0.7, 0.25, 0.0, 0.0, 0.01)), sample=8)


def test_non_finite_points_and_wide_thresholds(tiny):
    xyz = tiny.xyzB.copy()
    xyz[::7, 0] = np.nan
    xyz[1::11, 1] = np.inf
    xyz[2::13, 2] = -np.inf
    xyz[3::17] = 3e38
    spec = scangen.GridSpec(origin=(-20.0, -20.0, -1.0), res_m=1.0, dims=(40, 40, 8), feature=1, var_levels=5)
    etas = _lattice((4, 20, 2, 1, 1, 4), SMALL)
    _check(spec, tiny.xyzA, xyz, etas, var_thresh=[10, 100, 1000, 1 << 40])  # thresholds past 32 bits
    _check(spec, tiny.xyzA, xyz, etas, var_thresh=[0, 7, 7, 100000])


def test_dense_voxel_goes_to_the_exact_path():
    """70,000 points in one 0.5 m voxel: past the 32-bit sums, so its poses are redone exactly."""
    rng = np.random.default_rng(91)
    spec = scangen.lidar_grid(0.5)
    dense = np.stack([rng.uniform(a, a + 0.2, 70000) for a in (1.15, 2.15, 0.15)], 1)
    rest = np.stack([rng.uniform(-30, 30, 5000), rng.uniform(-30, 30, 5000), rng.uniform(-0.5, 5, 5000)], 1)
    xyz = np.concatenate([dense, rest]).astype(np.float32)
    redo = _check(spec, xyz, xyz, _lattice((2, 40, 2, 1, 1, 2), (0.05, 0.05, 0.05, 0.0, 0.0, 0.001)), sample=6)
    assert len(redo) > 0


@pytest.mark.parametrize("feature", [1, 2])
@pytest.mark.parametrize("n", [300, 1024, 3073, 8000])
def test_coarse_grids_redo_from_tiles(tiny, feature, n):
    """8 m voxels of hundreds of points: past the 32-bit sums (267), so poses are redone from the tiles
    that the groups' kernels wrote, at sizes around tiles and streams; one call with fewer points after
    one with more, and the same in a batch beside a pair for the table kernels, whose shape the tuner picks."""
    from paper_1709_06948_gb300 import align
    spec = scangen.GridSpec(origin=(-20.0, -20.0, -1.0), res_m=8.0, dims=(5, 5, 2), feature=feature, count_levels=7,
                            var_levels=8 if feature == 2 else 15)
    squeeze = np.array([0.05, 0.05, 1.0] if n < 8000 else [1.0, 1.0, 1.0], np.float32)  # dense at any size
    B = np.ascontiguousarray(tiny.xyzB[:n] * squeeze)
    etas = _lattice((4, 20, 2, 1, 1, 4), (6.0, 5.0, 0.3, 0.0, 0.0, 0.5))
    assert len(_check(spec, tiny.xyzA, B, etas)) > 0
    L, other = lib_grid(spec), lib_grid(tiny.grid)
    align.align_set_reference(L, tiny.xyzA)
    align.align_set_reference(other, tiny.xyzA)
    rng = np.random.default_rng(98)
    pairs = [(L, tiny.xyzB, etas), (other, tiny.xyzB, tiny.T + rng.uniform(-0.5, 0.5, (40, 6))), (L, B, etas)]
    b = align.align_batch_create()
    for tune in (False, True):
        got = align.align_eval_batch(b, pairs, tune=tune)
        for (mi, am), (G, xyz, e) in zip(got, pairs):
            align.align_set_sweep(G, 0)
            mi0, am0, _ = align.align_eval_mi(G, xyz, eta6=e)
            align.align_set_sweep(G, -1)
            assert np.array_equal(mi.view(np.int32), mi0.view(np.int32)) and am == am0
    align.align_batch_destroy(b)


def test_partition_count_stays_as_the_tables_left_it():
    """align_eval_stats' key partitions are the table kernels': neither groups whose redone poses need
    several (a voxel past the 32-bit sums, more voxels than a table holds) nor scattered poses change them."""
    from paper_1709_06948_gb300 import align
    rng = np.random.default_rng(97)
    spec = scangen.lidar_grid(0.5)
    dense = np.stack([rng.uniform(a, a + 0.2, 70000) for a in (1.15, 2.15, 0.15)], 1)
    rest = np.stack([rng.uniform(-39, 39, 60000), rng.uniform(-39, 39, 60000), rng.uniform(-0.9, 6.5, 60000)], 1)
    xyz = np.concatenate([dense, rest]).astype(np.float32)
    etas = _lattice((2, 40, 2, 1, 1, 2), (0.05, 0.05, 0.05, 0.0, 0.0, 0.001))
    L = lib_grid(spec)
    align.align_set_reference(L, xyz)

    def passes(kind, e):
        align.align_eval_mi(L, xyz, eta6=e)
        st = align.align_eval_stats(L)
        assert st["sweep"] == kind
        return st["passes"]
    assert passes(3, etas) == 1 and len(align.align_eval_redo_poses(L)) > 0
    align.align_set_sweep(L, 0)
    n = passes(0, etas[:40])
    assert n > 1
    align.align_set_sweep(L, -1)
    assert passes(4, etas[:1]) == n and passes(3, etas) == n
    L.close()


def test_not_a_lattice_keeps_the_table_kernels(tiny):
    """A pose missing, repeated or moved: not every combination, so the poses go to the tables."""
    etas = _lattice((4, 20, 2, 1, 1, 4), SMALL)
    moved = etas.copy()
    moved[17, 1] += 0.25
    for e in (etas[:-1], np.concatenate([etas[1:], etas[:1], etas[:1]]), moved):
        _check(tiny.grid, tiny.xyzA, tiny.xyzB, e, sweep=1)


@pytest.mark.parametrize("counts,sweep", [((2, 16, 2, 2, 2, 3), 1), ((2, 2, 2, 5, 5, 5), 1), ((8, 1, 2, 5, 5, 8), 1),
                                          ((4, 2, 2, 5, 5, 8), 1), ((3, 3, 2, 5, 5, 3), 3), ((5, 2, 2, 5, 5, 4), 3),
                                          ((3, 2, 8, 3, 3, 3), 3), ((8, 8, 1, 2, 2, 10), 3)])
def test_few_poses_per_list_keep_the_table_kernels(tiny, counts, sweep):
    """Lattices whose lists and groups serve few poses go to the tables from 2 groups per SM on."""
    _check(tiny.grid, tiny.xyzA, tiny.xyzB, _lattice(counts, SMALL), sweep=sweep, sample=8)


def test_search_levels_by_groups_equal_table_kernels():
    """The six-level search of a LiDAR pair: the same poses and MI with either kind of kernel."""
    from paper_1709_06948_gb300 import align
    pair = scangen.lidar_pair(seed=scangen.SEED_BASE + 95, n_beams=32)
    half = np.array([2.0, 2.0, 0.25, math.radians(1.0), math.radians(1.0), math.radians(5.0)])
    got = []
    for kind in (-1, 0):
        L = lib_grid(pair.grid)
        align.align_set_reference(L, pair.xyzA)
        align.align_set_sweep(L, kind)
        T, mi, lb = align.align_search(L, pair.xyzB, np.zeros(6), half, levels=6, counts=(8, 8, 2, 2, 2, 8))
        assert align.align_eval_stats(L)["sweep"] == (3 if kind < 0 else 0)
        got.append((T.tolist(), mi, lb.tolist()))
        L.close()
    assert got[0] == got[1]


@pytest.mark.parametrize("graph", [False, True])
def test_batch_mixes_groups_and_tables(tiny, graph):
    """Lattices of several grids and features beside pose sets that are none, in one batch (twice, the
    second with other poses): every pair's result is align_eval_mi's alone."""
    from paper_1709_06948_gb300 import align
    rng = np.random.default_rng(92)
    specs = [scangen.GridSpec(origin=(-20.0, -20.0, -1.0), res_m=r, dims=(int(40 / r), int(39 / r), int(8 / r)), feature=f,
                              count_levels=7, var_levels=8 if f == 2 else 15) for r, f in ((0.5, 2), (1.0, 1), (0.5, 0), (1.0, 2))]
    grids = []
    for spec in specs:
        L = lib_grid(spec)
        align.align_set_reference(L, tiny.xyzA)
        grids.append(L)
    b = align.align_batch_create()
    for shift in (0.0, 0.07):
        sets = [_lattice((3, 20, 2, 2, 1, 4), SMALL, centre=tiny.T + shift), _lattice((9, 13, 2, 2, 1, 3), SMALL, (0, 1, 2, 3, 4, 5)),
                tiny.T + rng.uniform(-0.5, 0.5, (40, 6)), _lattice((3, 20, 2, 2, 1, 4), SMALL, centre=tiny.T - shift)]
        pairs = [(L, tiny.xyzB[k::2], etas) for k, (L, etas) in enumerate(zip(grids, sets))]
        got = align.align_eval_batch(b, pairs, graph=graph)
        for (mi, am), (L, B, etas) in zip(got, pairs):
            align.align_set_sweep(L, 0)
            mi0, am0, _ = align.align_eval_mi(L, B, eta6=etas)
            align.align_set_sweep(L, -1)
            assert np.array_equal(mi.view(np.int32), mi0.view(np.int32)) and am == am0
    align.align_batch_destroy(b)


def test_batch_finds_lattices_after_other_pairs(tiny):
    """A lattice behind a pair without shared rotations goes by groups as it does before one: the same
    kernels, the same results; so does one whose rotations change fastest."""
    from paper_1709_06948_gb300 import align
    rng = np.random.default_rng(99)
    L = lib_grid(tiny.grid)
    align.align_set_reference(L, tiny.xyzA)
    other = tiny.T + rng.uniform(-0.5, 0.5, (40, 6))
    for order in ((3, 4, 5, 0, 1, 2), (0, 1, 2, 3, 4, 5)):
        lat = _lattice((8, 8, 2, 2, 2, 4), SMALL, order)
        seen = []
        for pairs in ([(L, tiny.xyzB, lat), (L, tiny.xyzB, other)], [(L, tiny.xyzB, other), (L, tiny.xyzB, lat)]):
            b = align.align_batch_create()
            got = align.align_eval_batch(b, pairs)
            k = 0 if pairs[0][2] is lat else 1
            seen.append((align.align_batch_stats(b)["kernel_launches"], got[k][0].tobytes(), got[k][1], got[1 - k][0].tobytes()))
            align.align_batch_destroy(b)
        assert seen[0] == seen[1] and seen[0][0] == 3 + 6 + 2  # pack, compose, argmax; groups' six, eval and redo
    L.close()
