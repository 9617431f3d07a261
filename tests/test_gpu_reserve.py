"""pf_reserve makes every later single-filter call of up to P_max particles free of
allocations: whole filter steps are captured in a graph right after it, on streams whose
workspace holds nothing else."""
import pytest

import oracle
from paper_1202_6163_gb300 import pf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("P", [1000, 16384, 16385, 100003, 1 << 20, (1 << 24) + 5])
def test_step_captured_right_after_reserve(P):
    g = torch.Generator(device="cuda")
    g.manual_seed(P)
    lw = torch.randn(P, device="cuda", generator=g)
    x = torch.randn(P, 2, device="cuda", generator=g)
    x0 = x.clone()
    anc, perm, metro = (torch.zeros(P, dtype=torch.int32, device="cuda") for _ in range(3))
    ess = torch.zeros(1, device="cuda")
    moved = torch.empty_like(x)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()  # a workspace of its own
    with torch.cuda.stream(stream):
        pf.pf_reserve(P, 0, 0)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            pf.pf_ess(lw, P, ess)
            pf.pf_resample_metropolis(lw, P, 2, 1, metro)
            for resample in (pf.pf_resample_multinomial, pf.pf_resample_stratified, pf.pf_resample_systematic):
                resample(lw, P, 0, 7, anc)
            pf.pf_gather(x, P, 8, anc, P, moved)
            pf.pf_permute(anc, P, perm)
            pf.pf_gather_inplace(x, P, 8, perm)
        graph.replay()
        assert pf.pf_get_device_status() == pf.PF_OK
    assert torch.equal(moved, x0[anc.long()]) and torch.equal(x, x0[perm.long()])
    if P <= 100003:
        assert (perm.cpu().numpy() == oracle.permute(anc.cpu().numpy())).all()
    assert float(ess) > 1.0
