"""The tile scan at its branches: threads whose weights are all positive and threads
with zero weights among them, at every number of elements per thread (4, 8, 16), on
tiles that end inside a thread's share and that begin with an alignment lead.  Every
decision is compared with the FP64 oracle under the near-tie rule."""
import numpy as np
import pytest

import oracle
from paper_1202_6163_gb300 import pf
from parity import check_cumulative

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def zero_runs(P, pattern, seed):
    """N(0,1) log-weights with zero weights: single ones, a whole thread's share and
    its neighbours, the tail, or weights 2^-60 of the rest (sums near the fixed point's end)."""
    rng = np.random.default_rng(seed)
    lw = rng.standard_normal(P).astype(np.float32)
    if pattern == "single":
        lw[rng.random(P) < 0.05] = -np.inf
    elif pattern == "shares":
        for at in range(0, P, 97):
            lw[at:at + 33] = -np.inf
    elif pattern == "tail":
        lw[P - P // 3:] = -np.inf
    elif pattern == "tiny":
        lw[rng.random(P) < 0.7] -= 41.0
    lw[P // 2] = 0.5
    return lw


@pytest.mark.parametrize("pattern", ["none", "single", "shares", "tail", "tiny"])
@pytest.mark.parametrize("P,lead", [(2045, 3), (8193, 0), (1300007, 1), (2500013, 2)])
def test_scan_branches_match_oracle(P, lead, pattern):
    lw = zero_runs(P, pattern, seed=P + lead)
    buf = torch.empty(P + lead, device="cuda")
    buf[lead:] = torch.from_numpy(lw).cuda()
    anc = torch.empty(P, dtype=torch.int32, device="cuda")
    pf.pf_resample_systematic(buf[lead:], P, 0, 11, anc)
    assert pf.pf_get_device_status() == pf.PF_OK
    rep = check_cumulative("systematic", lw, anc.cpu().numpy(), oracle.systematic(lw, 11), 11)
    assert rep.ok, rep.summary()
