"""Filters of one tile per CTA beyond a cluster's: CTA counts on either side of the
change from polled records to the arrival counter and up to the resident CTAs, the
calls of other kinds in between that share the arrival counters, a withheld record under
both ways of waiting, and domain errors.  Against the FP64 oracle under the near-tie
rule."""
import numpy as np
import pytest

import oracle
from paper_1202_6163_gb300 import pf
from parity import check_cumulative

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KINDS = {"systematic": (pf.pf_resample_systematic, oracle.systematic),
         "stratified": (pf.pf_resample_stratified, oracle.stratified)}
SIZES = [32769, 2048 * 40, 2048 * 40 + 1, 2048 * 41 + 3, 622592, 622593, 1300001, 2490368, 2490369]


def one(name, lw, d, seed):
    P = lw.size
    anc = torch.full((P,), -3, dtype=torch.int32, device="cuda")
    KINDS[name][0](d, P, 0, seed, anc)
    assert pf.pf_get_device_status() == pf.PF_OK
    rep = check_cumulative(name, lw, anc.cpu().numpy(), KINDS[name][1](lw, seed), seed)
    assert rep.ok, (P, rep.summary())


@pytest.mark.parametrize("name", list(KINDS))
@pytest.mark.parametrize("P", SIZES)
def test_cta_counts(name, P):
    lw = (2.0 * np.random.default_rng(P).standard_normal(P)).astype(np.float32)
    lw[P // 4:P // 4 + 9000] = -np.inf  # CTAs without mass among the records
    d = torch.from_numpy(lw).cuda()
    one(name, lw, d, 3)
    multi = torch.empty(P, dtype=torch.int32, device="cuda")
    pf.pf_resample_multinomial(d, P, 0, 1, multi)  # two arrivals, its own records
    one(name, lw, d, 4)


@pytest.mark.parametrize("name", list(KINDS))
@pytest.mark.parametrize("P", [40000, 500000])
def test_withheld_record_and_domain(name, P):
    lw = np.random.default_rng(1).standard_normal(P).astype(np.float32)
    d = torch.from_numpy(lw).cuda()
    anc = torch.empty(P, dtype=torch.int32, device="cuda")
    try:
        pf.pf_set_wait_limit_ns(2_000_000)
        pf.pf_debug_skip_publish(5)
        KINDS[name][0](d, P, 0, 3, anc)
        assert pf.pf_get_device_status() == pf.PF_ERR_TIMEOUT
    finally:
        pf.pf_set_wait_limit_ns(1_000_000_000)
        pf.pf_debug_skip_publish(-1)
    one(name, lw, d, 6)
    for bad in (float("nan"), float("inf")):
        e = d.clone()
        e[P - 3] = bad
        KINDS[name][0](e, P, 0, 3, anc)
        assert pf.pf_get_device_status() == pf.PF_ERR_DOMAIN
    KINDS[name][0](torch.full_like(d, -float("inf")), P, 0, 3, anc)
    assert pf.pf_get_device_status() == pf.PF_ERR_DOMAIN
    one(name, lw, d, 7)
