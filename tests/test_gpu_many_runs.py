"""More long runs in one tile than the CTA-wide decode stores ahead (128): those left over
go through its chunks, whichever they are.  Compared with the FP64 oracle under the near-tie
rule; the entries around the ancestors must stay untouched."""
import numpy as np
import pytest

import oracle
from paper_1202_6163_gb300 import pf
from parity import check_cumulative

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KINDS = {"systematic": (pf.pf_resample_systematic, oracle.systematic),
         "stratified": (pf.pf_resample_stratified, oracle.stratified)}


@pytest.mark.parametrize("name", list(KINDS))
@pytest.mark.parametrize("runs, spread", [(127, 0.0), (129, 0.0), (300, 0.0), (300, 0.3)])
def test_equally_heavy_neighbours(name, runs, spread):
    """`runs` neighbours with about 10400 to 26000 offspring each among 4 million particles."""
    fn, orc = KINDS[name]
    P, at = 4000003, 1234567
    rng = np.random.default_rng(runs)
    lw = rng.standard_normal(P).astype(np.float32)
    heavy = np.exp(spread * rng.standard_normal(runs))
    lw[at:at + runs] = -np.inf
    share = 0.8 if runs >= 300 else 0.5
    rest = np.exp(lw.astype(np.float64)).sum()
    lw[at:at + runs] = np.log(heavy / heavy.sum() * rest * share / (1 - share))
    d = torch.from_numpy(lw).cuda()
    ref = orc(lw, 11)
    for shift in (0, 3):
        buf = torch.full((P + 8,), -3, dtype=torch.int32, device="cuda")
        fn(d, P, 0, 11, buf[shift:])
        assert pf.pf_get_device_status() == pf.PF_OK
        got = buf.cpu().numpy()
        assert (got[:shift] == -3).all() and (got[shift + P:] == -3).all()
        rep = check_cumulative(name, lw, got[shift:shift + P], ref, 11)
        assert rep.ok, rep.summary()
