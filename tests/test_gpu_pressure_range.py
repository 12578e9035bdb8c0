"""Pressure forces at the ends of the FP32 range: pairs far closer than 1e-15 in
systems of that scale, and pressures that overflow only in terms that are 0 (a
particle with itself, coincident particles).  Against the oracle, 1e-5 of the sum
of the pair forces as in the other pass tests."""
import numpy as np
import pytest

import oracle as orc
from paper_2602_19873_gb300 import nl

from nlcheck import TILES, gpu_build, oracle_sorted

pytestmark = pytest.mark.gpu
F = np.float32
SHAPES = [(m, j, 0) for m, j in TILES] + [(m, m, 1) for m in (4, 8, 16)]


def check(p, h, m, pres, cluster, jcl, half, periodic=0):
    import torch
    p = np.asarray(p, F)
    n = len(p)
    lo = np.full(3, -20 * h, F)
    box = {"lo": lo, "hi": -lo, "periodic": np.full(3, periodic, np.int32)}
    d = {"x": p[:, 0].copy(), "y": p[:, 1].copy(), "z": p[:, 2].copy(), "h": np.full(n, h, F),
         "m": np.full(n, m, F), "box": box, "kind": 1, "support": 2.0}
    o = oracle_sorted(d)
    rows = np.arange(n)
    off, idx = orc.brute_neighbors(o["xs"], o["ys"], o["zs"], o["hs"], box, 2.0, 1, rows)
    pr, rho = np.full(n, pres, F), np.ones(n, F)
    *want, fa = orc.sph_force(o["xs"], o["ys"], o["zs"], o["hs"], o["ms"], rho, pr, box, off, idx, rows)
    L, t = gpu_build(d, cluster=cluster, j_cluster=jcl, half_list=half)
    out = [torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(3)]
    L.force_pass(nl.NL_FORCE_SPH_PRESSURE, *out, m=t["m"], rho=torch.from_numpy(rho).cuda(),
                 pres=torch.from_numpy(pr).cuda())
    got = np.stack([a.cpu().numpy()[o["perm"]] for a in out], 1)
    L.free()
    assert fa.max() > 0
    err = np.linalg.norm(got - np.stack(want, 1), axis=1) / np.maximum(fa, 1e-300)
    assert np.all(err[fa > 0] <= 1e-5), err
    assert np.all(got[fa == 0] == 0)


@pytest.mark.parametrize("cluster,jcl,half", SHAPES)
@pytest.mark.parametrize("h,r", [(1e-9, 1e-16), (1e-11, 1e-18), (5e-12, 3e-19), (1e-11, 1e-20)])
def test_pairs_at_any_distance_have_their_own_kernel_gradient(h, r, cluster, jcl, half):
    check([(0.0, 0.0, 0.0), (0.6 * r, 0.0, 0.8 * r)], h, 1.0, 1e-30, cluster, jcl, half)


@pytest.mark.parametrize("cluster,jcl,half", SHAPES)
@pytest.mark.parametrize("periodic", [0, 1])
def test_terms_that_are_zero_stay_zero_where_pressures_are_large(periodic, cluster, jcl, half):
    """Pairs at 1.3 h and beyond, two of the particles coincident: their forces
    are finite, 2 P / h is not."""
    p = [(0.0, 0.0, 0.0), (1.3, 0.0, 0.0), (0.0, 1.4, 0.0), (0.0, 0.0, -1.5), (0.0, 0.0, -1.5)]
    check(p, 1.0, 1e-10, 2.5e38, cluster, jcl, half, periodic)


@pytest.mark.parametrize("cluster,jcl,half", SHAPES)
def test_coincident_particles_of_large_mass(cluster, jcl, half):
    """m 2C/h overflows, the mass of the particles within range times their
    coefficients does not."""
    p = [(0.0, 0.0, 0.0), (1.3, 0.0, 0.0), (0.0, 0.0, -1.5), (0.0, 0.0, -1.5)]
    check(p, 1.0, 1e30, 2.2e8, cluster, jcl, half)


@pytest.mark.parametrize("cluster,jcl,half", SHAPES)
def test_coefficients_that_overflow_where_forces_do_not(cluster, jcl, half):
    """3 P / (pi rho^2 h^4) is beyond FP32, its products with w' at 1.5 h are not."""
    p = [(0.0, 0.0, 0.0), (0.75, 0.0, 0.0), (0.0, 0.8, 0.0), (0.0, 0.0, -0.85)]
    check(p, 0.5, 1e-10, 2.6e37, cluster, jcl, half)
