"""The packed pass kernel at its edges: sizes around which one, two, four or
eight warps share a super-cluster, ragged last super-clusters, every tile shape
it serves, periodic systems whose entries wrap, inputs that are not finite, and
a support for which the scalar kernel runs instead.  Against the FP64 oracle
with the tolerances of the other pass tests (density 1e-5, forces 1e-5 of the
sum of the pair forces, counts exact)."""
import numpy as np
import pytest

import oracle as orc
from paper_2602_19873_gb300 import nl
from paper_2602_19873_gb300 import workloads as wl

from nlcheck import DENSITY_RTOL, full_reference, gpu_build, gpu_counts, gpu_density, oracle_sorted

pytestmark = pytest.mark.gpu
FORCE_RTOL = 1e-5


def _density(o, d, g_off, g_idx, ms=None):
    return orc.density(o["xs"], o["ys"], o["zs"], o["hs"], o["ms"] if ms is None else ms, d["box"],
                       g_off, g_idx, np.arange(len(o["xs"])))


# super-clusters of 64 particles: 1, and on both sides of 304, 608 and 1216
# (152 SMs x 16 warp slots / 8, 4, 2)
@pytest.mark.parametrize("n", [5, 63, 64, 65, 200, 304 * 64, 304 * 64 + 1, 608 * 64 - 5, 608 * 64 + 3,
                               1216 * 64, 1216 * 64 + 7])
@pytest.mark.parametrize("half", [0, 1])
def test_density_and_counts_around_the_split_sizes(n, half):
    d = wl.uniform(n, seed=300 + n % 97, n_target=min(30.0, 0.3 * n))
    o = oracle_sorted(d)
    g_off, g_idx = orc.gather_all(o["xs"], o["ys"], o["zs"], o["hs"], d["box"], d["support"])
    L, t = gpu_build(d, half_list=half)
    assert np.array_equal(gpu_counts(L, n)[o["perm"]], np.diff(g_off))
    want = _density(o, d, g_off, g_idx)
    rel = np.abs(gpu_density(L, t, n)[o["perm"]] - want) / want
    assert rel.max() <= DENSITY_RTOL, rel.max()
    L.free()


@pytest.mark.parametrize("n", [800, 19457, 39001])
@pytest.mark.parametrize("cluster,jcl,half", [(8, 8, 0), (8, 8, 1), (16, 16, 0), (16, 16, 1), (16, 8, 0)])
def test_lj_force_around_the_split_sizes(n, cluster, jcl, half):
    import torch
    d = wl.lj_fluid(n, seed=310 + n % 89, rc=0.55)
    o = oracle_sorted(d)
    g_off, g_idx = orc.gather_all(o["xs"], o["ys"], o["zs"], o["hs"], d["box"], d["support"])
    fx, fy, fz, fa = orc.lj_force(o["xs"], o["ys"], o["zs"], d["box"], 1.0, 0.3, g_off, g_idx, np.arange(n))
    L, t = gpu_build(d, cluster=cluster, j_cluster=jcl, half_list=half)
    out = [torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(3)]
    L.force_pass(nl.NL_FORCE_LJ, *out, eps=1.0, sigma=0.3)
    torch.cuda.synchronize()
    got = np.stack([a.cpu().numpy()[o["perm"]] for a in out], 1)
    err = np.linalg.norm(got - np.stack([fx, fy, fz], 1), axis=1) / np.maximum(fa, 1e-300)
    assert err[fa > 0].max() <= FORCE_RTOL, err[fa > 0].max()
    assert np.all(got[fa == 0] == 0)
    L.free()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("cluster,jcl", [(8, 8), (16, 8), (16, 16)])
def test_a_mass_that_is_not_finite_reaches_its_neighbors_only(cluster, jcl, bad):
    """Full lists: the particles without the marked one in their range keep
    their densities."""
    d = dict(wl.evrard(6000, seed=320, n_target=40.0))
    o = oracle_sorted(d)
    g_off, g_idx, _, _ = full_reference(o, d)
    n = len(o["xs"])
    mark = 1234
    m = d["m"].copy()
    m[o["perm"][mark]] = bad
    d["m"] = m
    L, t = gpu_build(d, cluster=cluster, j_cluster=jcl)
    got = gpu_density(L, t, n)[o["perm"]]
    near = np.zeros(n, bool)
    near[mark] = True
    for i in range(n):
        near[i] |= mark in g_idx[g_off[i]:g_off[i + 1]]
    assert near.sum() > 5
    want = _density(o, d, g_off, g_idx)
    rel = np.abs(got[~near] - want[~near]) / want[~near]
    assert rel.max() <= DENSITY_RTOL, rel.max()
    assert not np.isfinite(got[mark])
    L.free()


@pytest.mark.parametrize("half", [0, 1])
@pytest.mark.parametrize("support", [1.5, 1.0])
def test_a_support_below_the_kernels_sums_its_own_pairs(support, half):
    """r = support h below 2h: the pairs beyond r take no part (the range test
    of the scalar kernel)."""
    d = dict(wl.evrard(5000, seed=330, n_target=60.0))
    d["support"] = support
    o = oracle_sorted(d)
    g_off, g_idx, _, _ = full_reference(o, d)
    n = len(o["xs"])
    L, t = gpu_build(d, half_list=half)
    want = _density(o, d, g_off, g_idx)
    rel = np.abs(gpu_density(L, t, n)[o["perm"]] - want) / want
    assert rel.max() <= DENSITY_RTOL, rel.max()
    L.free()


@pytest.mark.parametrize("n", [900, 39001])
@pytest.mark.parametrize("cluster,half", [(8, 0), (8, 1), (16, 0), (16, 1)])
def test_lj_forces_overflow_where_their_coefficient_does(n, cluster, half):
    """Pairs at 7e-4: 24 eps (2 s^12 - s^6) / r^2 exceeds FP32 (3.6e39), the force
    itself (2.6e36) would not; at 1e-3 (2.5e37) it is finite."""
    import torch
    d = wl.lj_fluid(n, seed=330 + n % 89, rc=0.55)
    for k, r in ((0, 7e-4), (2, 1e-3)):
        for a in "xyz":
            d[a][k] = np.float32(0.001 + 0.2 * k)
            d[a][k + 1] = np.float32(d[a][k] + r / np.sqrt(3.0))
    L, t = gpu_build(d, cluster=cluster, j_cluster=cluster, half_list=half)
    out = [torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(3)]
    L.force_pass(nl.NL_FORCE_LJ, *out, eps=1.0, sigma=0.3)
    got = np.stack([a.cpu().numpy() for a in out], 1)
    assert np.all(got[0] == -np.inf) and np.all(got[1] == np.inf)
    x = [np.array([d[a][k] for a in "xyz"], np.float64) for k in (2, 3)]
    dv = x[1] - x[0]
    r2 = dv @ dv
    s6 = (0.09 / r2) ** 3
    f = 24.0 / r2 * s6 * (2 * s6 - 1) * dv
    assert np.allclose(got[3], f, rtol=1e-5) and np.allclose(got[2], -f, rtol=1e-5)
    assert np.isfinite(got[2:]).all()
    L.free()
