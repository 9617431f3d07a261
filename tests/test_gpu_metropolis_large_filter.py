"""Batched Metropolis filters beyond the 2^17 particles at which a cumulative one stops: they
run like any other, beside small ones.  Filter 0 with key s is the single call with seed s, bit
for bit; sampled chains of every filter against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_1202_6163_gb300 import pf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("B", [8, -1])
@pytest.mark.parametrize("sizes", [(200003, 300), (131072, 131073, 131074, 5), (1 << 20,)])
def test_filters_beyond_the_cumulative_limit(sizes, B):
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    g = torch.Generator(device="cuda")
    g.manual_seed(len(sizes))
    lw = 0.3 * torch.randn(int(off[-1]), device="cuda", generator=g)
    seeds = np.arange(40, 40 + len(sizes), dtype=np.uint64)
    anc = torch.full((int(off[-1]) + 1,), -3, dtype=torch.int32, device="cuda")
    chosen = torch.zeros(len(sizes), dtype=torch.int32, device="cuda")
    args = (lw, torch.from_numpy(off).cuda(), len(sizes))
    keys = torch.from_numpy(seeds.view(np.int64)).cuda()
    if B >= 0:
        pf.pf_resample_batched(pf.PF_METROPOLIS, *args, B, keys, anc)
        steps = [B] * len(sizes)
    else:
        pf.pf_resample_batched_metropolis_bound(*args, 0.1, keys, anc, chosen)
        steps = chosen.cpu().tolist()
    assert pf.pf_get_device_status() == pf.PF_OK
    assert int(anc[-1]) == -3 and min(steps) > 0
    alone = torch.empty(sizes[0], dtype=torch.int32, device="cuda")
    pf.pf_resample_metropolis(lw[:sizes[0]], sizes[0], steps[0], int(seeds[0]), alone)
    assert torch.equal(anc[:sizes[0]], alone)
    host, got = lw.cpu().numpy(), anc.cpu().numpy()
    for f, n in enumerate(sizes):
        part = host[off[f]:off[f + 1]]
        idx = np.unique(np.linspace(0, n - 1, 500).astype(np.int64))
        ref = oracle.metropolis(part, steps[f], int(seeds[f]), f, chains=idx)
        # a chain differs only where a decision's uniform lies within 1e-6 of its ratio
        assert (got[off[f]:off[f + 1]][idx] != ref).sum() <= 1
