"""The initial draw at the state widths with a variant of their own (16) and without one
(12, 64): several groups of four normals per particle, ragged last blocks.  Against the
oracle, with the tolerance of the widths tested beside the step: a few ulps of the mean and
of sqrt(p0) |z|."""
import numpy as np
import pytest

import oracle
from paper_1202_6163_gb300 import pf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("F,P,D", [(3, 1025, 12), (2, 5003, 16), (2, 300, 64), (1, 3, 16)])
def test_init_widths(F, P, D):
    x = torch.full((F * P * D + 8,), 9.0, device="cuda")
    lw = torch.full((F, P), 7.0, device="cuda")
    ll, ls = (torch.full((F,), 3.0, dtype=torch.float64, device="cuda") for _ in range(2))
    es = torch.zeros(F, device="cuda")
    rs = torch.ones(F, dtype=torch.int32, device="cuda")
    pf.pf_lg_init(F, P, D, 0.5, 2.0, 41, x, lw, ll, ls, es, rs)
    assert pf.pf_get_device_status() == pf.PF_OK
    got = x.cpu().numpy()
    assert (got[F * P * D:] == 9.0).all()
    np.testing.assert_allclose(got[:F * P * D].reshape(F, P, D), oracle.lg_init(F, P, D, 0.5, 2.0, 41)["x"],
                               rtol=2e-6, atol=4e-6)
    assert (lw.cpu().numpy() == 0).all() and (rs.cpu().numpy() == 0).all()
