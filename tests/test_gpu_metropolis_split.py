"""Batched Metropolis filters around the limits of the shared-memory staging: whole
(57344 weights), split between shared and global memory (up to 114688) and read from L2
beyond; step counts that end inside a group of draws; weights that underflow, for
which a step decides on the log-weights.  Both chain streams, against the FP64
oracle under the near-tie rule."""
import numpy as np
import pytest

import oracle
from paper_1202_6163_gb300 import pf
from parity import check_metropolis

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = [57344, 57345, 65536, 114688, 114689, 1023]


@pytest.mark.parametrize("spread", [1.0, 60.0])  # 60: most weights far below 2^-100 of the largest
@pytest.mark.parametrize("B", [1, 7, 32])
def test_staging_limits(B, spread):
    rng = np.random.default_rng(B)
    off = np.zeros(len(SIZES) + 1, np.int64)
    np.cumsum(SIZES, out=off[1:])
    lw = (spread * rng.standard_normal(int(off[-1]))).astype(np.float32)
    lw[rng.random(lw.size) < 0.01] = -np.inf
    seeds = np.arange(50, 50 + len(SIZES), dtype=np.uint64)
    anc = torch.full((lw.size,), -3, dtype=torch.int32, device="cuda")
    pf.pf_resample_batched(pf.PF_METROPOLIS, torch.from_numpy(lw).cuda(), torch.from_numpy(off).cuda(), len(SIZES), B,
                           torch.from_numpy(seeds.view(np.int64)).cuda(), anc)
    assert pf.pf_get_device_status() == pf.PF_OK
    got = anc.cpu().numpy()
    for f, P in enumerate(SIZES):
        part = lw[off[f]:off[f + 1]]
        idx = np.unique(rng.integers(0, P, size=min(P, 4000)))
        ref = oracle.metropolis(part, B, int(seeds[f]), f, chains=idx)
        rep = check_metropolis(part, B, got[off[f]:off[f + 1]][idx], ref, int(seeds[f]), chains=idx, filter_id=f)
        assert rep.ok, (P, rep.summary())
