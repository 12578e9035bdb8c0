"""Records of the batched search where its batches, node chunks and particle
tests have their edges: leaves longer than one batch of j-clusters (piles of
coincident particles at the deepest octree level), super-clusters far wider
than their radii (sparse halos around a dense core, tested particle by
particle), systems of one particle to a few super-clusters, and leaf buckets
that give trees of one node up to thousands.  Byte for byte against the
oracle's canonical lists, for every tile shape, full and half, open and
periodic."""
import numpy as np
import pytest

from nlcheck import TILES, compare_records, full_reference, gpu_build, oracle_sorted

pytestmark = pytest.mark.gpu
F = np.float32


def _system(pos, h, periodic, kind=1, lo=0.0):
    pos = np.ascontiguousarray(pos, F)
    box = {"lo": np.full(3, lo, F), "hi": np.full(3, lo + 1.0, F), "periodic": np.full(3, periodic, np.int32)}
    n = len(pos)
    return {"x": pos[:, 0].copy(), "y": pos[:, 1].copy(), "z": pos[:, 2].copy(),
            "h": np.ascontiguousarray(h, F), "m": np.ones(n, F), "box": box, "kind": kind, "support": 2.0}


def piles(periodic):
    """Two piles of coincident particles and a thin uniform background."""
    rng = np.random.default_rng(31)
    p = np.concatenate([np.full((700, 3), 0.2), np.full((333, 3), 0.7), rng.random((600, 3)) * 0.999])
    h = np.concatenate([np.full(1033, 0.01), rng.uniform(0.02, 0.06, 600)])
    return _system(p, h, periodic)


def halo(periodic):
    """A dense core with small radii inside a sparse halo whose radii differ
    by a factor of twenty."""
    rng = np.random.default_rng(32)
    core = 0.5 + 0.01 * rng.normal(size=(2000, 3))
    out = rng.random((400, 3)) * 0.999
    h = np.concatenate([np.full(2000, 0.0012), rng.uniform(0.005, 0.1, 400)])
    return _system(np.concatenate([core, out]), h, periodic)


def cloud(n, periodic):
    rng = np.random.default_rng(n)
    return _system(rng.random((n, 3)) * 0.999, rng.uniform(0.03, 0.08, n), periodic)


def _check(d, tile, half, bucket=256, compress=1):
    M, MJ = tile
    if half and M != MJ:
        pytest.skip("half lists have j-clusters of the i-cluster size")
    o = oracle_sorted(d)
    _, _, p_off, p_idx = full_reference(o, d)
    L, _ = gpu_build(d, cluster=M, j_cluster=MJ, half_list=half, bucket=bucket, compress=compress)
    nsc = L.sizes()["n_superclusters"]
    compare_records(L, o, d, M, compress, np.arange(nsc), np.arange(len(o["xs"])), p_off, p_idx,
                    jcluster=MJ, half=bool(half))
    L.free()


@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("half", [0, 1])
@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("make", [piles, halo])
def test_long_leaves_and_wide_superclusters(make, tile, half, periodic):
    _check(make(periodic), tile, half)


@pytest.mark.parametrize("bucket", [8, 1024])
@pytest.mark.parametrize("periodic", [0, 1])
def test_deep_and_shallow_trees(bucket, periodic):
    _check(halo(periodic), (8, 8), 1, bucket)
    _check(cloud(3000, periodic), (8, 8), 0, bucket)


@pytest.mark.parametrize("half", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 31, 63, 64, 65, 129, 511, 2047])
def test_small_systems(n, half):
    for tile in ((8, 8), (4, 4), (16, 16)):
        _check(cloud(n, n % 2), tile, half)


def lattice(scale, periodic):
    """Spacings and ranges that differ by a few ulps: the fused sums of the tile
    test cannot decide these pairs, which need the canonical predicate; at the
    small scale squared distances are denormal."""
    rng = np.random.default_rng(33)
    m = 12
    g = (np.indices((m, m, m)).reshape(3, -1).T + 0.5) / m
    p = g * (1 + rng.integers(-3, 4, g.shape) * 6e-8)
    h = (1 + rng.integers(-3, 4, len(g)) * 6e-8) / (2 * m)
    return _system(scale * p, scale * h, periodic)


@pytest.mark.parametrize("half", [0, 1])
@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("scale,periodic", [(1.0, 0), (1.0, 1), (3e-21, 0)])
def test_pairs_at_the_edge_of_the_range(scale, periodic, tile, half):
    _check(lattice(scale, periodic), tile, half)


@pytest.mark.parametrize("lo", [-0.5, 3.0, 1024.0])
@pytest.mark.parametrize("half", [0, 1])
def test_periodic_boxes_off_the_origin(lo, half):
    """Images of particles round to the size of the coordinates: far from the
    origin the differences are wrapped one by one instead."""
    rng = np.random.default_rng(35)
    d = _system(lo + rng.random((6000, 3)) * 0.999, rng.uniform(0.02, 0.05, 6000), 1, lo=lo)
    for tile in ((8, 8), (4, 4), (16, 16)):
        _check(d, tile, half)
