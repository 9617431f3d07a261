"""Filters beyond one cooperative launch (P > 2^25) whose last tile is ragged and holds a
particle with tens of thousands of offspring: the tile's weights are read back, and its last
warp has lanes past the end beside strata far from the tile's first.  Compared with the FP64
oracle under the near-tie rule; the entries around the ancestors must stay untouched."""
import numpy as np
import pytest

import oracle
from paper_1202_6163_gb300 import pf
from parity import check_cumulative

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TILE = 8192


# (elements of the last tile, the heavy one among them, its offspring)
@pytest.mark.parametrize("tail, at, offspring", [(4153, 0, 30000), (4153, 4150, 20000), (TILE - 1, 700, 60000)])
def test_heavy_particle_in_a_ragged_last_tile(tail, at, offspring):
    P = (1 << 25) + tail
    lw = np.random.default_rng(tail + at).standard_normal(P, dtype=np.float32)
    place = (1 << 25) + at
    lw[place] = -np.inf
    lw[place] = np.log(np.exp(lw, dtype=np.float64).sum() * offspring / (P - offspring))
    buf = torch.full((P + 2,), -3, dtype=torch.int32, device="cuda")
    pf.pf_resample_stratified(torch.from_numpy(lw).cuda(), P, 0, 5, buf[1:])
    assert pf.pf_get_device_status() == pf.PF_OK
    got = buf.cpu().numpy()
    assert got[0] == -3 and got[-1] == -3
    assert abs(int((got[1:-1] == place).sum()) - offspring) <= 2
    rep = check_cumulative("stratified", lw, got[1:-1], oracle.stratified(lw, 5), 5)
    assert rep.ok, rep.summary()
