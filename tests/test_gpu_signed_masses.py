"""Density sums of inputs of both signs: half lists give the sums of full lists.
Against the oracle, 1e-5 of the sum of the absolute terms."""
import numpy as np
import pytest

import oracle as orc
from paper_2602_19873_gb300 import workloads as wl

from nlcheck import DENSITY_RTOL, full_reference, gpu_build, gpu_density, oracle_sorted

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cluster,half", [(8, 0), (16, 0), (4, 1), (8, 1), (16, 1)])
@pytest.mark.parametrize("name,support", [("evrard", 2.0), ("uniform", 2.0), ("evrard", 1.5)])
def test_density_of_signed_inputs(name, support, cluster, half):
    d = dict(wl.evrard(3001, seed=341, n_target=40.0) if name == "evrard" else wl.uniform(3001, seed=342, n_target=40.0))
    n = len(d["x"])
    d["support"] = support
    d["m"] = (d["m"] * np.random.default_rng(343).choice([-1.0, 1.0], n)).astype(np.float32)
    o = oracle_sorted(d)
    g_off, g_idx, _, _ = full_reference(o, d)
    rho = lambda m: orc.density(o["xs"], o["ys"], o["zs"], o["hs"], m, d["box"], g_off, g_idx, np.arange(n))
    L, t = gpu_build(d, cluster=cluster, half_list=half)
    err = np.abs(gpu_density(L, t, n)[o["perm"]] - rho(o["ms"])) / rho(np.abs(o["ms"]))
    assert err.max() <= DENSITY_RTOL, err.max()
    L.free()
