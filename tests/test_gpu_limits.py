"""The largest particle counts the entry points accept, where 32-bit index arithmetic has no
room left: the calls run to the end and every entry is right."""
import pytest

from paper_1202_6163_gb300 import pf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

P_MAX = 2147483647  # PF_MAX_PARTICLES


@pytest.mark.parametrize("P", [P_MAX, P_MAX - 8192])
def test_permute_all_offspring_of_one_particle(P):
    """Every tile but one is empty slots; one tile lists P - 1 extra copies."""
    kept = 1234567890
    a = torch.full((P,), kept, dtype=torch.int32, device="cuda")
    out = torch.full((P + 1,), -3, dtype=torch.int32, device="cuda")
    pf.pf_permute(a, P, out)
    assert pf.pf_get_device_status() == pf.PF_OK
    assert bool(torch.equal(out[:P], a)) and int(out[P]) == -3


@pytest.mark.parametrize("name", ["systematic", "stratified"])
def test_one_particle_takes_every_offset(name):
    """All other weights are zero: one run of P offspring from one tile."""
    kept = 1234567890
    lw = torch.full((P_MAX,), float("-inf"), device="cuda")
    lw[kept] = 0.5
    out = torch.full((P_MAX + 2,), -3, dtype=torch.int32, device="cuda")
    getattr(pf, "pf_resample_" + name)(lw, P_MAX, 0, 3, out[1:])
    assert pf.pf_get_device_status() == pf.PF_OK
    assert bool((out[1:-1] == kept).all()) and int(out[0]) == -3 and int(out[-1]) == -3


def test_rows_of_more_than_2_to_32_chunks():
    """17 GB to a row, aligned to 4 bytes only: a chunk's place in its row takes 33 bits."""
    n = (1 << 32) + 5
    x = torch.zeros(2 * n, dtype=torch.int32, device="cuda")
    for lo in range(0, n, 1 << 30):  # row 0 counts; row 1 is zero
        hi = min(n, lo + (1 << 30))
        x[lo:hi] = torch.arange(lo - (1 << 31), hi - (1 << 31), dtype=torch.int64, device="cuda").to(torch.int32)
    out = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    zero = torch.zeros(2, dtype=torch.int32, device="cuda")
    pf.pf_gather(x, 2, 4 * n, zero, 1, out)
    assert torch.equal(out[:n], x[:n]) and int(out[n]) == 0
    del out
    pf.pf_gather_inplace(x, 2, 4 * n, zero)
    assert pf.pf_get_device_status() == pf.PF_OK
    assert torch.equal(x[:n], x[n:])
