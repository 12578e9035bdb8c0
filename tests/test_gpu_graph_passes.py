"""Passes on a list between replays of its graph: a replay finds the buffers that
it was captured with, whatever other passes ran in between."""
import numpy as np
import pytest

from paper_2602_19873_gb300 import nl
from paper_2602_19873_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cluster,half", [(8, 0), (8, 1), (16, 1), (4, 0)])
def test_replays_after_other_passes(cluster, half):
    import torch
    stream = torch.cuda.Stream()
    systems = wl.batched(n_systems=5, seed=531, log_n=(2.7, 3.7))
    offs = np.concatenate([[0], np.cumsum([len(d["x"]) for d in systems])]).astype(np.int64)
    n = int(offs[-1])
    dev = {k: torch.from_numpy(np.concatenate([d[k] for d in systems]).astype(np.float32)).cuda() for k in "xyzhm"}
    boxes = [d["box"] for d in systems]
    p = nl.make_params(key=1, cluster=cluster, support=2.0, half_list=half)
    with torch.cuda.stream(stream):
        rho, out = torch.zeros(n, device="cuda"), [torch.empty(n, device="cuda") for _ in range(3)]
        L = nl.NeighborList()
        G = nl.Graph(L, dev["x"], dev["y"], dev["z"], dev["h"], dev["m"], rho, offs, boxes, p, stream)
        G.launch(stream)
        G.check(stream)
        want = rho.clone()
        pres = want * want
        counts = torch.empty(n, dtype=torch.int32, device="cuda")
        others = (lambda: L.force_pass(nl.NL_FORCE_SPH_PRESSURE, *out, m=dev["m"], rho=want, pres=pres, stream=stream),
                  lambda: L.force_pass(nl.NL_FORCE_LJ, *out, eps=1.0, sigma=1e-3, stream=stream),
                  lambda: L.force_pass(nl.NL_FORCE_LJ_COULOMB, *out, m=dev["m"], eps=1.0, sigma=1e-3, stream=stream),
                  lambda: L.nearest_distance(out[0], stream),
                  lambda: L.neighbor_counts(counts, stream))
        for other in others:
            other()
            taken = [torch.full((n, k), 7.0, device="cuda") for k in (2, 4)]  # what was freed is in use again
            rho.zero_()
            G.launch(stream)
            G.check(stream)
            assert torch.equal(rho, want)
            del taken
        stream.synchronize()
        G.free()
        L.free()
