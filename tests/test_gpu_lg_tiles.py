"""The initial draw on either side of the count of tiles from which a CTA takes 1024
particles instead of 256, at state widths with a variant of their own and without one.
Against the oracle, with the tolerance of the other widths' test; the entries behind the
states stay untouched."""
import numpy as np
import pytest

import oracle
from paper_1202_6163_gb300 import pf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("F,P,D", [(151, 1024, 4), (152, 1024, 4), (303, 1024, 4), (2, 310001, 4), (5, 70001, 20), (400, 257, 64),
                                   (151, 2047, 8), (310, 1000, 16), (1, 255, 32)])
def test_init_tiles(F, P, D):
    x = torch.full((F * P * D + 8,), 9.0, device="cuda")
    lw = torch.full((F * P + 1,), 7.0, device="cuda")
    ll, ls = (torch.full((F,), 3.0, dtype=torch.float64, device="cuda") for _ in range(2))
    es = torch.zeros(F, device="cuda")
    rs = torch.ones(F, dtype=torch.int32, device="cuda")
    pf.pf_lg_init(F, P, D, 0.5, 2.0, 41, x, lw, ll, ls, es, rs)
    assert pf.pf_get_device_status() == pf.PF_OK
    got = x.cpu().numpy()
    assert (got[F * P * D:] == 9.0).all()
    np.testing.assert_allclose(got[:F * P * D].reshape(F, P, D), oracle.lg_init(F, P, D, 0.5, 2.0, 41)["x"],
                               rtol=2e-6, atol=4e-6)
    assert (lw[:-1] == 0).all() and float(lw[-1]) == 7.0
    assert (ll == 0).all() and (rs == 0).all() and (es == P).all()
