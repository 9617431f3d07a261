"""Batched systematic and stratified calls on either side of the change from filters split
over CTAs to whole ones: the route is no part of the result, so a call whose filters are
kept whole writes what the same filters give in masked calls that split them; and
one-tile filters of every width beside them.  Sampled filters against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1202_6163_gb300 import pf
from parity import check_cumulative

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KINDS = {"systematic": (pf.PF_SYSTEMATIC, oracle.systematic), "stratified": (pf.PF_STRATIFIED, oracle.stratified)}


@pytest.mark.parametrize("name", list(KINDS))
@pytest.mark.parametrize("P", [8190, 20001])  # two tiles where the filter starts off the 16-byte grid, three
@pytest.mark.parametrize("beyond", [-1, 0, 1, 40])
def test_route_is_no_part_of_the_result(name, P, beyond):
    kind, orc = KINDS[name]
    grid = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    sizes = [P] * (3 * grid // 4 + beyond) + [1, 3, 2045, 2048, 2049, 4096, 4097, 8192, 8189]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    F = len(sizes)
    lw = (2.0 * np.random.default_rng(P + beyond).standard_normal(off[-1])).astype(np.float32)
    d = torch.from_numpy(lw).cuda()
    o = torch.from_numpy(off).cuda()
    seeds = torch.arange(F, dtype=torch.int64, device="cuda") * 7
    a = torch.full((lw.size,), -9, dtype=torch.int32, device="cuda")
    b = torch.full_like(a, -9)
    pf.pf_resample_batched(kind, d, o, F, 0, seeds, a)
    for r in range(4):
        mask = (torch.arange(F, device="cuda") % 4 == r).to(torch.int32)
        pf.pf_resample_batched_masked(kind, d, o, F, 0, seeds, mask, b)
    assert pf.pf_get_device_status() == pf.PF_OK
    assert torch.equal(a, b)
    anc = a.cpu().numpy()
    for f in [0, 1, 2, F - 10] + list(range(F - 9, F)):
        l = lw[off[f]:off[f + 1]]
        rep = check_cumulative(name, l, anc[off[f]:off[f + 1]], orc(l, 7 * f, f), 7 * f, filter_id=f)
        assert rep.ok, (f, l.size, rep.summary())
