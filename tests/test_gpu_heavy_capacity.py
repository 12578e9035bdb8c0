"""Full lists of systems in which most super-clusters are heavy (every particle
reaches every other): the half search learns in a few rounds how many upper
entries and tuples there are, from whatever room it starts with."""
import numpy as np
import pytest

import oracle as orc
from paper_2602_19873_gb300 import nl

from nlcheck import gpu_counts, gpu_records

pytestmark = pytest.mark.gpu
F = np.float32


# (more than three super-clusters per resident block: fewer are not set aside)
@pytest.mark.parametrize("n,blocks,cap0", [(120002, 0, None), (40010, 1, None), (40010, 1, 0), (40010, 1, 100000)])
@pytest.mark.parametrize("periodic", [0, 1])
def test_every_list_holds_the_whole_system(n, blocks, cap0, periodic, monkeypatch):
    import torch
    if cap0 is not None:
        monkeypatch.setenv("NLGB_HALF_CAP0", str(cap0))
    rng = np.random.default_rng(n)
    # (a periodic box wide enough for a radius that holds the cube)
    p = torch.from_numpy((rng.random((3, n)) * 0.999).astype(F)).cuda()
    box = {"lo": np.full(3, -2.0, F), "hi": np.full(3, 2.0, F), "periodic": np.full(3, periodic, np.int32)}
    h = torch.full((n,), 0.9, device="cuda")
    L = nl.NeighborList().build(p[0].contiguous(), p[1].contiguous(), p[2].contiguous(), h, box,
                                nl.make_params(key=1, support=2.0, blocks_per_sm=blocks))
    ncl, nsc = -(-n // 8), -(-n // 64)
    whole = orc.encode_record(np.arange(ncl, dtype=np.uint32), np.full(ncl, 0xff, np.uint32), 32, True)
    last = orc.encode_record(np.arange(ncl, dtype=np.uint32),
                             np.full(ncl, (1 << (ncl - 8 * (nsc - 1))) - 1, np.uint32), 32, True)
    for s, (at, cnt, data) in zip((0, nsc // 2, nsc - 2, nsc - 1), gpu_records(L, (0, nsc // 2, nsc - 2, nsc - 1))):
        want = last if s == nsc - 1 else whole
        assert cnt == ncl and np.array_equal(data[at:at + len(want)], want)
    assert L.sizes()["n_entries"] == ncl * nsc
    assert np.all(gpu_counts(L, n) == n - 1)
    L.free()
