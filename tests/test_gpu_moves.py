"""The in-place permutation and the two row moves at the edges of their kernels: tile
ends, tiles whose extra copies fill several parts of the listing, unaligned outputs,
and rows of every chunk width (4 to 32 bytes, powers of two and not) at bases aligned
to less than the chunk.  Bit for bit the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1202_6163_gb300 import pf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def ancestors(P, law, seed):
    rng = np.random.default_rng(seed)
    if law == "sorted":
        a = np.sort(rng.integers(0, P, P))
    elif law == "random":
        a = rng.integers(0, P, P)
    elif law == "one":
        a = np.full(P, P - 1)
    else:  # a few particles with runs longer than a part, the rest single
        a = np.arange(P)
        for f in range(3):
            lo = f * P // 3
            a[lo:lo + P // 4] = min(lo + P // 8, P - 1)
    return a.astype(np.int32)


@pytest.mark.parametrize("law", ["sorted", "random", "one", "runs"])
@pytest.mark.parametrize("P", [1, 31, 4095, 4096, 4097, 8193, 100003])
def test_permute_edges(P, law):
    a = ancestors(P, law, seed=P)
    for shift in (0, 1):
        out = torch.full((P + 2,), -3, dtype=torch.int32, device="cuda")
        pf.pf_permute(torch.from_numpy(a).cuda(), P, out[shift:])
        assert pf.pf_get_device_status() == pf.PF_OK
        got = out.cpu().numpy()
        assert np.array_equal(got[shift:shift + P], oracle.permute(a))
        assert (got[:shift] == -3).all() and (got[shift + P:] == -3).all()


@pytest.mark.parametrize("dim", [1, 2, 3, 4, 5, 6, 8, 12, 16, 24, 40])
@pytest.mark.parametrize("shift", [0, 4, 1])  # floats past a 256-byte boundary
def test_row_moves(dim, shift):
    P = 5003
    a = ancestors(P, "random", seed=dim)
    perm = oracle.permute(a)
    x = np.random.default_rng(dim).standard_normal((P, dim)).astype(np.float32)
    src = torch.empty(P * dim + shift, device="cuda")
    src[shift:] = torch.from_numpy(x.reshape(-1)).cuda()
    for P_dst in (P, 1777):
        dst = torch.full((P_dst * dim + shift + 1,), -3.0, device="cuda")
        pf.pf_gather(src[shift:], P, 4 * dim, torch.from_numpy(a).cuda(), P_dst, dst[shift:])
        got = dst.cpu().numpy()
        assert np.array_equal(got[shift:-1].reshape(P_dst, dim), x[a[:P_dst]])
        assert (got[:shift] == -3).all() and got[-1] == -3
    pf.pf_gather_inplace(src[shift:], P, 4 * dim, torch.from_numpy(perm).cuda())
    assert pf.pf_get_device_status() == pf.PF_OK
    assert np.array_equal(src[shift:].cpu().numpy().reshape(P, dim), x[perm])


def test_bad_rows_are_left_and_reported():
    P, dim = 3000, 8
    a = np.arange(P, dtype=np.int32)
    a[7], a[2999], a[100], a[101] = P, -1, 101, 102  # out of range; a source that does not keep its slot
    x = torch.arange(P * dim, dtype=torch.float32, device="cuda").reshape(P, dim)
    before = x.clone()
    pf.pf_gather_inplace(x, P, 4 * dim, torch.from_numpy(a).cuda())
    assert pf.pf_get_device_status() == pf.PF_ERR_INVALID
    want = before.clone()
    want[101] = before[102]
    assert torch.equal(x, want)


@pytest.mark.parametrize("dim", [1, 3, 24, 32])
def test_waves_of_several_pieces(dim):
    """More chunks than one resident wave takes at once, so that every CTA goes on to further
    pieces with their entries asked for early; odd sizes leave a ragged last piece."""
    P = 1000003
    g = torch.Generator(device="cuda")
    g.manual_seed(dim)
    lw = 2.0 * torch.randn(P, device="cuda", generator=g)
    a = torch.empty(P, dtype=torch.int32, device="cuda")
    perm = torch.empty_like(a)
    pf.pf_resample_systematic(lw, P, 0, 3, a)
    pf.pf_permute(a, P, perm)
    x = torch.randn(P, dim, device="cuda", generator=g)
    ref = x[perm.long()]
    out = torch.empty_like(x)
    pf.pf_gather(x, P, 4 * dim, a, P, out)
    assert torch.equal(out, x[a.long()])
    pf.pf_gather_inplace(x, P, 4 * dim, perm)
    assert pf.pf_get_device_status() == pf.PF_OK
    assert torch.equal(x, ref)


@pytest.mark.parametrize("law", ["sorted", "random", "one", "runs"])
@pytest.mark.parametrize("P", [2, 32, 1023, 1024, 1025, 12321, 16383, 16384, 16385])
def test_permute_in_one_cta(P, law):
    """Either side of the count up to which one CTA forms the permutation, and where its
    threads' shares of the particles end unevenly."""
    a = ancestors(P, law, seed=P)
    out = torch.full((P + 2,), -3, dtype=torch.int32, device="cuda")
    pf.pf_permute(torch.from_numpy(a).cuda(), P, out[1:])
    assert pf.pf_get_device_status() == pf.PF_OK
    got = out.cpu().numpy()
    assert np.array_equal(got[1:P + 1], oracle.permute(a)) and got[0] == -3 and got[-1] == -3
