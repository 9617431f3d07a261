"""Single filters of up to 16 tiles, which one thread-block cluster resamples: every
number of tiles around the cluster sizes, unaligned slices, tiles of every width (a
minimum tile of 8192 makes them full), counts that one tile owns alone, domain
errors, and the ancestors of a filter one tile past the cluster's.  Against the
FP64 oracle under the near-tie rule."""
import numpy as np
import pytest

import oracle
from paper_1202_6163_gb300 import pf
from parity import check_cumulative

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KINDS = {"systematic": (pf.PF_SYSTEMATIC, pf.pf_resample_systematic, oracle.systematic),
         "stratified": (pf.PF_STRATIFIED, pf.pf_resample_stratified, oracle.stratified),
         "multinomial": (pf.PF_MULTINOMIAL, pf.pf_resample_multinomial, oracle.multinomial)}


def run(name, lw, seed, lead=0, shift=0):
    _, fn, _ = KINDS[name]
    P = lw.size
    buf = torch.empty(P + lead, device="cuda")
    buf[lead:] = torch.from_numpy(lw).cuda()
    out = torch.full((P + 8,), -3, dtype=torch.int32, device="cuda")
    fn(buf[lead:], P, 0, seed, out[shift:])
    got = out.cpu().numpy()
    assert (got[:shift] == -3).all() and (got[shift + P:] == -3).all()
    return got[shift:shift + P]


def check(name, lw, got, seed):
    assert pf.pf_get_device_status() == pf.PF_OK
    rep = check_cumulative(name, lw, got, KINDS[name][2](lw, seed), seed)
    assert rep.ok, (lw.size, rep.summary())


@pytest.mark.parametrize("name", list(KINDS))
@pytest.mark.parametrize("P", [1, 2, 3, 7, 511, 2048, 2049, 4097, 8193, 16384, 16385, 18433, 32765, 32768, 32769])
def test_tiles_of_a_cluster(name, P):
    rng = np.random.default_rng(P)
    for lead, shift, spread in ((0, 0, 1.0), (3, 1, 4.0), (1, 2, 0.25)):
        lw = (spread * rng.standard_normal(P)).astype(np.float32)
        check(name, lw, run(name, lw, 9 + lead, lead, shift), 9 + lead)


@pytest.mark.parametrize("name", list(KINDS))
def test_zero_weights_and_one_owner(name):
    for P in (1500, 20011, 32768):
        lw = np.random.default_rng(P).standard_normal(P).astype(np.float32)
        lw[P // 3:P // 3 + 5000] = -np.inf  # tiles without weight
        lw[::7] = -np.inf
        check(name, lw, run(name, lw, 4), 4)
        lw[:] = -np.inf
        lw[P - 1] = 2.0  # one tile owns every offset
        check(name, lw, run(name, lw, 5), 5)


@pytest.mark.parametrize("name", list(KINDS))
@pytest.mark.parametrize("P", [8190, 8193, 40000, 131069, 131073])
def test_full_tiles(name, P):
    kind = KINDS[name][0]
    try:
        pf.pf_set_min_tile(kind, P, 8192)
        lw = (2.0 * np.random.default_rng(P).standard_normal(P)).astype(np.float32)
        check(name, lw, run(name, lw, 6, lead=2), 6)
    finally:
        pf.pf_set_min_tile(kind, P, 0)


@pytest.mark.parametrize("name", list(KINDS))
@pytest.mark.parametrize("P", [1000, 20011])
def test_domain_errors(name, P):
    for bad in (np.nan, np.inf, None):
        lw = np.zeros(P, np.float32)
        if bad is None:
            lw[:] = -np.inf
        else:
            lw[P - 2] = bad
        run(name, lw, 1)
        assert pf.pf_get_device_status() == pf.PF_ERR_DOMAIN
    lw = np.zeros(P, np.float32)
    check(name, lw, run(name, lw, 2), 2)
