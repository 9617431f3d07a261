"""Many calls back to back on one stream, each reading what the one before it wrote into the
same buffers, with no synchronisation between: a call may start up while the work before it
still runs, and must see all that it wrote.  Every pass's results are compared with the same
calls made one at a time."""
import pytest

from paper_1202_6163_gb300 import pf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PASSES = 24


def chain(P, dim, seed, apart):
    """PASSES filter steps on one set of buffers; each pass's results, read through pf_gather."""
    def done():
        if apart:
            torch.cuda.synchronize()

    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    table = 2.0 * torch.randn(4 * P, device="cuda", generator=g)
    picks = [torch.randint(0, 4 * P, (P,), dtype=torch.int32, device="cuda", generator=g) for _ in range(PASSES)]
    every = torch.arange(P, dtype=torch.int32, device="cuda")
    x = torch.randn(P, dim, device="cuda", generator=g)
    y, lw = torch.empty_like(x), torch.empty(P, device="cuda")
    anc, perm, metro = (torch.zeros(P, dtype=torch.int32, device="cuda") for _ in range(3))
    ess = torch.zeros(PASSES, device="cuda")
    kept = [[torch.empty(P, dtype=torch.int32, device="cuda") for _ in range(3)] +
            [torch.empty(P, dim, device="cuda") for _ in range(2)] for _ in range(PASSES)]
    torch.cuda.synchronize()
    kinds = [pf.pf_resample_systematic, pf.pf_resample_multinomial, pf.pf_resample_stratified]
    for t in range(PASSES):
        calls = [lambda: pf.pf_gather(table, 4 * P, 4, picks[t], P, lw),  # this pass's log-weights
                 lambda: pf.pf_ess(lw, P, ess[t:]),
                 lambda: kinds[t % 3](lw, P, 0, t, anc),
                 lambda: pf.pf_gather(x, P, 4 * dim, anc, P, y),
                 lambda: pf.pf_permute(anc, P, perm),
                 lambda: pf.pf_gather_inplace(x, P, 4 * dim, perm),
                 lambda: pf.pf_resample_metropolis(lw, P, -1 if P < 3000 else 5, t, metro)]
        calls += [lambda a=a, b=b, w=w: pf.pf_gather(a, P, w, every, P, b)
                  for a, b, w in zip((anc, perm, metro, x, y), kept[t], (4, 4, 4, 4 * dim, 4 * dim))]
        for call in calls:
            call()
            done()
    assert pf.pf_get_device_status() == pf.PF_OK
    return kept, ess


@pytest.mark.parametrize("P, dim", [(100, 3), (1000, 4), (2049, 1), (20011, 8), (65536, 4), (300007, 5)])
def test_chained_calls(P, dim):
    one_at_a_time, ess1 = chain(P, dim, seed=P, apart=True)
    for _ in range(3):
        got, ess = chain(P, dim, seed=P, apart=False)
        for t in range(PASSES):
            for name, a, b in zip(("ancestors", "permuted", "metropolis", "states", "gathered"), got[t], one_at_a_time[t]):
                assert torch.equal(a, b), (t, name)
        assert torch.equal(ess, ess1)
