"""The padding slots of a system's last super-cluster take part in nothing,
wherever the particles lie and however large their radii are: counts, nearest
distances, Lennard-Jones and Lennard-Jones + Coulomb forces of a few particles in
boxes far from the origin, of the size of the FP32 range, and periodic, and with
radii whose squares overflow.  Against the oracle (counts exact, distances 1e-6,
forces 1e-5 of the sum of the pair forces, as in the other pass tests)."""
import numpy as np
import pytest

import oracle as orc
from paper_2602_19873_gb300 import nl

from nlcheck import TILES, gpu_build, gpu_counts, oracle_sorted

pytestmark = pytest.mark.gpu
F = np.float32

# name: box, corner and edge of the cube that holds the particles, h
PLACES = {
    "far": ((0.0, 2e18), 0, 1e18, 1e17, 4e16),
    "far below": ((-2e18, 0.0), 0, -1e18, 1e17, 4e16),
    "radius": ((0.0, 1.0), 0, 0.0, 1.0, 1e19),
    "whole range": ((-1.6e38, 1.6e38), 0, -0.5, 1.0, 0.3),
    "end of the range": ((1e38, 3e38), 0, 1e38, 2e37, 1e37),
    "periodic": ((0.0, 1e18), 1, 0.0, 0.9999e18, 1.2e17),
    "periodic, radius": ((0.0, 1e33), 1, 0.0, 0.9999e33, 1.2e32),
}


def system(place, n):
    (lo, hi), per, corner, edge, h = PLACES[place]
    rng = np.random.default_rng(n)
    p = (corner + edge * rng.random((n, 3))).astype(F)
    box = {"lo": np.full(3, lo, F), "hi": np.full(3, hi, F), "periodic": np.full(3, per, np.int32)}
    return {"x": p[:, 0].copy(), "y": p[:, 1].copy(), "z": p[:, 2].copy(), "h": np.full(n, h, F),
            "m": rng.choice([-1.0, 1.0], n).astype(F), "box": box, "kind": 1, "support": 2.0}, edge


@pytest.mark.parametrize("cluster,jcl,half", [(m, j, 0) for m, j in TILES] + [(m, m, 1) for m in (4, 8, 16)])
@pytest.mark.parametrize("n", [5, 70])
@pytest.mark.parametrize("place", list(PLACES))
def test_padding_takes_part_in_nothing(place, n, cluster, jcl, half):
    import torch
    d, edge = system(place, n)
    o = oracle_sorted(d)
    rows = np.arange(n)
    off, idx = orc.brute_neighbors(o["xs"], o["ys"], o["zs"], o["hs"], d["box"], 2.0, 0, rows)
    L, t = gpu_build(d, cluster=cluster, j_cluster=jcl, half_list=half)
    assert np.array_equal(gpu_counts(L, n)[o["perm"]], np.diff(off))
    out = [torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(3)]
    L.nearest_distance(out[0])
    got = out[0].cpu().numpy()[o["perm"]]
    want = orc.nearest(o["xs"], o["ys"], o["zs"], d["box"], off, idx)
    fin = np.isfinite(want)
    # (a distance whose FP32 square overflows is infinite)
    fin &= want < 1.8e19
    assert np.array_equal(np.isfinite(got), fin)
    assert np.all(np.abs(got[fin] - want[fin]) <= 1e-6 * want[fin])
    if edge > 1e30:  # pair forces overflow or vanish: no particle has a neighbor here
        assert len(idx) == 0
    sigma = 0.1 * edge
    for kind, kw, ref in (
            (nl.NL_FORCE_LJ, {}, orc.lj_force(o["xs"], o["ys"], o["zs"], d["box"], 1.0, sigma, off, idx, rows)),
            (nl.NL_FORCE_LJ_COULOMB, {"m": t["m"], "kc": 1.0},
             orc.ljc_force(o["xs"], o["ys"], o["zs"], d["box"], 1.0, sigma, o["ms"], 1.0, off, idx, rows))):
        L.force_pass(kind, *out, eps=1.0, sigma=sigma, **kw)
        f = np.stack([a.cpu().numpy()[o["perm"]] for a in out], 1)
        fa = ref[3]
        err = np.linalg.norm(f - np.stack(ref[:3], 1), axis=1) / np.maximum(fa, 1e-300)
        assert np.all(f[fa == 0] == 0)
        assert np.all(err[fa > 0] <= 1e-5), err.max()
    L.free()
