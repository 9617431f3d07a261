"""The permutation's passes over tiles of 4096 slots, which serve more than 16384 particles:
tile ends, more tiles than the last CTA scans in one round of 512, tiles split into parts, and
an ancestor out of range.  Bit for bit the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1202_6163_gb300 import pf
from test_gpu_moves import ancestors

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("law", ["sorted", "random", "one", "runs"])
@pytest.mark.parametrize("P", [5 * 4096 - 1, 5 * 4096, 5 * 4096 + 1, 512 * 4096 + 1, 2 * 512 * 4096 + 4097])
def test_tile_ends_and_rounds(P, law):
    a = ancestors(P, law, seed=P)
    for shift in (0, 1):
        out = torch.full((P + 2,), -3, dtype=torch.int32, device="cuda")
        pf.pf_permute(torch.from_numpy(a).cuda(), P, out[shift:])
        assert pf.pf_get_device_status() == pf.PF_OK
        got = out.cpu().numpy()
        assert np.array_equal(got[shift:shift + P], oracle.permute(a))
        assert (got[:shift] == -3).all() and (got[shift + P:] == -3).all()


@pytest.mark.parametrize("bad", [-1, 40000, -2147483648, 2147483647])
def test_ancestor_out_of_range(bad):
    P = 40000
    a = ancestors(P, "random", seed=1)
    a[12345] = bad
    out = torch.full((P + 1,), -3, dtype=torch.int32, device="cuda")
    pf.pf_permute(torch.from_numpy(a).cuda(), P, out)
    assert pf.pf_get_device_status() == pf.PF_ERR_INVALID
    assert int(out[P]) == -3
