"""A mixed plan with more items than a grid's z dimension holds pairs of."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")


def test_plan_of_33000_bins():
    n, N, Nb = 33000, 6, 2
    g = torch.Generator(device="cuda").manual_seed(1)
    Q = torch.randn((n, Nb, N), dtype=torch.complex64, device="cuda", generator=g)
    b = pg.BatchedSVD([Q[i].t() for i in range(n)], kmodes=1)
    b.run()
    assert b.status() == pg.OK
    S = torch.linalg.svdvals(Q.to(torch.complex128).cpu())
    got = b.S_all.cpu().reshape(n, Nb)
    # binary32 inputs, exact products: an M eps_32 backward error at most
    assert torch.all(torch.abs(got - S) <= Nb * 2.0 ** -24 * S[:, :1])
