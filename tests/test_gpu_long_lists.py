"""Super-clusters whose lists are far longer than the others': a few particles
whose radii reach most of a system.  Their search is split into parts and their
lists are shared by many warps in the passes; records must be the oracle's byte
for byte, counts and nearest distances the oracle's, densities and forces within
the tolerances of the other pass tests.  The sizes put their lists above one
block's share (8192 entries) in the largest system."""
import numpy as np
import pytest

import oracle as orc
from paper_2602_19873_gb300 import nl

from nlcheck import DENSITY_RTOL, compare_records, full_reference, gpu_build, gpu_counts, gpu_density, oracle_sorted

pytestmark = pytest.mark.gpu
F = np.float32


def giants(n, periodic, n_giants=5):
    rng = np.random.default_rng(n)
    p = (rng.random((n, 3)) * 0.9999).astype(F)
    h = np.full(n, 0.5 * (3.0 * 20.0 / (4.0 * np.pi * n)) ** (1.0 / 3.0), F)
    big = rng.choice(n, n_giants, replace=False)
    h[big] = rng.uniform(0.22, 0.245, n_giants) if periodic else rng.uniform(0.3, 0.9, n_giants)
    box = {"lo": np.zeros(3, F), "hi": np.ones(3, F), "periodic": np.full(3, periodic, np.int32)}
    return {"x": p[:, 0].copy(), "y": p[:, 1].copy(), "z": p[:, 2].copy(), "h": h.astype(F),
            "m": rng.uniform(0.5, 1.5, n).astype(F) / n, "box": box, "kind": 1, "support": 2.0}


@pytest.fixture(scope="module")
def cases():
    out = {}
    for name, n, per in (("open", 80007, 0), ("periodic", 60013, 1)):
        d = giants(n, per)
        o = oracle_sorted(d)
        out[name] = (d, o, full_reference(o, d))
    return out


@pytest.mark.parametrize("half", [0, 1])
@pytest.mark.parametrize("cluster", [8, 16, 4])
@pytest.mark.parametrize("name", ["open", "periodic"])
def test_records_and_passes(cases, name, cluster, half):
    import torch
    d, o, (g_off, g_idx, p_off, p_idx) = cases[name]
    n = len(o["xs"])
    L, t = gpu_build(d, cluster=cluster, half_list=half)
    nsc = L.sizes()["n_superclusters"]
    total, so, J, m = compare_records(L, o, d, cluster, 1, np.arange(nsc), np.arange(n), p_off, p_idx,
                                      half=bool(half))
    if not half:  # (how much of a giant's list a half list keeps depends on its place)
        assert np.diff(so).max() > (8192 if name == "open" and cluster == 8 else 1024)
    assert L.sizes()["n_entries"] == len(J)
    assert np.array_equal(gpu_counts(L, n)[o["perm"]], np.diff(g_off))
    want = orc.density(o["xs"], o["ys"], o["zs"], o["hs"], o["ms"], d["box"], g_off, g_idx, np.arange(n))
    rel = np.abs(gpu_density(L, t, n)[o["perm"]] - want) / want
    assert rel.max() <= DENSITY_RTOL, rel.max()
    dist = torch.empty(n, dtype=torch.float32, device="cuda")
    L.nearest_distance(dist)
    near = orc.nearest(o["xs"], o["ys"], o["zs"], d["box"], g_off, g_idx)
    got = dist.cpu().numpy()[o["perm"]]
    fin = np.isfinite(near)
    assert np.array_equal(np.isfinite(got), fin)
    assert (np.abs(got[fin] - near[fin]) / near[fin]).max() <= 1e-6
    out = [torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(3)]
    L.force_pass(nl.NL_FORCE_LJ, *out, eps=1.0, sigma=0.001)
    fx, fy, fz, fa = orc.lj_force(o["xs"], o["ys"], o["zs"], d["box"], 1.0, 0.001, g_off, g_idx, np.arange(n))
    f = np.stack([a.cpu().numpy()[o["perm"]] for a in out], 1)
    err = np.linalg.norm(f - np.stack([fx, fy, fz], 1), axis=1) / np.maximum(fa, 1e-300)
    assert err[fa > 0].max() <= 1e-5, err[fa > 0].max()
    L.free()


def test_h_iteration_from_lists_of_whole_systems():
    """A start whose first lists hold most of the system converges to counts in
    the window, checked by the oracle."""
    import torch
    d = giants(30011, 0, n_giants=40)
    t = {k: torch.from_numpy(d[k]).cuda() for k in ("x", "y", "z", "h")}
    L = nl.NeighborList()
    p = nl.make_params(key=1, support=2.0)
    info = L.iterate_h(t["x"], t["y"], t["z"], t["h"], d["box"], p, 60, tol=2.0, start=nl.NL_HSTART_GIVEN)
    assert info["unconverged"] == 0
    rows = np.arange(0, 30011, 97)
    cnt = orc.gather_counts_brute(d["x"], d["y"], d["z"], t["h"].cpu().numpy(), d["box"], 2.0, rows)
    assert np.abs(np.asarray(cnt) - 60).max() <= 2
    L.free()
