"""The warp-by-warp assignment at its branches: warps whose offsets take one staging
chunk or several, tiles on either side of the count that sends them to the CTA-wide
decode, every alignment of the ancestors, and whole filters whose last tile has fewer
elements per thread than the others (the CTA's warps are then in tiles of different
widths at the same time).  Compared with the FP64 oracle under the near-tie rule; the
entries around the ancestors must stay untouched."""
import numpy as np
import pytest

import oracle
from paper_1202_6163_gb300 import pf
from parity import check_cumulative

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KINDS = {"systematic": (pf.PF_SYSTEMATIC, pf.pf_resample_systematic, oracle.systematic),
         "stratified": (pf.PF_STRATIFIED, pf.pf_resample_stratified, oracle.stratified)}


@pytest.mark.parametrize("name", list(KINDS))
@pytest.mark.parametrize("share", [0.002, 0.02, 0.3, 0.409, 0.41, 0.9])
def test_dominant_particle(name, share):
    """One particle with `share` of the weight: 80 to 36000 of 40000 offsets in one warp."""
    _, fn, orc = KINDS[name]
    P = 40000
    lw = np.random.default_rng(3).standard_normal(P).astype(np.float32)
    w = np.exp(lw.astype(np.float64))
    at = 12345
    lw[at] = np.log(share / (1 - share) * (w.sum() - w[at]))
    d = torch.from_numpy(lw).cuda()
    ref = orc(lw, 7)
    for shift in range(4):
        buf = torch.full((P + 8,), -3, dtype=torch.int32, device="cuda")
        fn(d, P, 0, 7, buf[shift:])
        assert pf.pf_get_device_status() == pf.PF_OK
        got = buf.cpu().numpy()
        assert (got[:shift] == -3).all() and (got[shift + P:] == -3).all()
        rep = check_cumulative(name, lw, got[shift:shift + P], ref, 7)
        assert rep.ok, rep.summary()


@pytest.mark.parametrize("name", list(KINDS))
def test_whole_filters_of_mixed_widths(name):
    kind, _, orc = KINDS[name]
    rng = np.random.default_rng(5)
    sizes = np.array([8192 * (1 + i % 3) + (100, 1500, 3000, 7000)[i % 4] for i in range(640)], dtype=np.int64)
    off = np.zeros(sizes.size + 1, np.int64)
    np.cumsum(sizes, out=off[1:])
    lw = rng.standard_normal(int(off[-1]))
    lw[rng.random(lw.size) < 0.01] += 10.0  # a warp's share runs from none of the tile's offsets to most
    lw = lw.astype(np.float32)
    seeds = np.arange(100, 100 + sizes.size, dtype=np.uint64)
    anc = torch.full((lw.size,), -3, dtype=torch.int32, device="cuda")
    pf.pf_resample_batched(kind, torch.from_numpy(lw).cuda(), torch.from_numpy(off).cuda(), sizes.size, 0,
                           torch.from_numpy(seeds.view(np.int64)).cuda(), anc)
    assert pf.pf_get_device_status() == pf.PF_OK
    got = anc.cpu().numpy()
    for f in range(0, sizes.size, 5):
        part = lw[off[f]:off[f + 1]]
        rep = check_cumulative(name, part, got[off[f]:off[f + 1]], orc(part, int(seeds[f]), f), int(seeds[f]),
                               filter_id=f)
        assert rep.ok, (f, rep.summary())


@pytest.mark.parametrize("name", list(KINDS))
@pytest.mark.parametrize("runs", [(1279,), (1280, 1281), (640, 5000, 3), (65000,), (30000, 36000), (20479, 20480, 41000),
                                  (150000, 9000)])
def test_long_runs(name, runs):
    """Neighbouring particles with long runs (some in one thread, some across threads), in
    tiles on either side of the 65536 offsets that send a tile to the CTA-wide decode, with
    particles of a few offsets around them and zero weights between: the runs stored as they
    are, and the chunks between them, at every alignment."""
    _, fn, orc = KINDS[name]
    P = 300000
    lw = np.random.default_rng(len(runs)).standard_normal(P).astype(np.float32)
    lw[70001:70010:3] = -np.inf
    places = [70002, 70003, 70035][:len(runs)]
    lw[places] = -np.inf
    rest = np.exp(lw.astype(np.float64)).sum()
    total = rest * P / (P - sum(runs))
    lw[places] = np.log(np.array(runs) / P * total)
    lw[70300:70400] = np.log(30.0 * total / P)  # a warp of many middling runs
    d = torch.from_numpy(lw).cuda()
    ref = orc(lw, 11)
    for shift in range(4):
        buf = torch.full((P + 8,), -3, dtype=torch.int32, device="cuda")
        fn(d, P, 0, 11, buf[shift:])
        assert pf.pf_get_device_status() == pf.PF_OK
        got = buf.cpu().numpy()
        assert (got[:shift] == -3).all() and (got[shift + P:] == -3).all()
        rep = check_cumulative(name, lw, got[shift:shift + P], ref, 11)
        assert rep.ok, rep.summary()
