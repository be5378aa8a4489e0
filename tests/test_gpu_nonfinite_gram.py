"""Infinities and NaN on the Gram route: cotangents of pod_backward, and a
working copy that overflows, come out as NaN and not as some number."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("where", ["dU", "dS", "dVT"])
def test_nonfinite_cotangents(where, bad, prec):
    N, M = 1500, 20
    rng = np.random.default_rng(1)
    X = rng.standard_normal((N, M)) * 2.0 ** -np.arange(M)
    X = torch.from_numpy(np.ascontiguousarray(X.T)).cuda().to(torch.float32 if prec else torch.float64).t()
    out = []
    for b in (0, 500):
        f = pg.pod(X, remove_mean=False, r_max=3, prec=prec, leaf_rows=b)
        g = torch.Generator(device="cuda").manual_seed(1)
        c = dict(dU=torch.randn((f.r, N), dtype=torch.float64, device="cuda", generator=g).t(),
                 dS=torch.randn(M, dtype=torch.float64, device="cuda", generator=g),
                 dVT=torch.randn((M, M), dtype=torch.float64, device="cuda", generator=g))
        c["dS"][3:] = 0.0
        if where == "dS":
            c[where][1] = bad
        else:
            c[where][2, 1] = bad
        out.append(pg.pod_backward(f, (N, M), None, False, 0, b, 3, **c))
    finite = torch.isfinite(out[1])
    assert not finite.all()
    assert not torch.isfinite(out[0])[~finite].any()


def test_working_copy_that_overflows():
    X = np.random.default_rng(2).standard_normal((900, 14))
    X[5, 3] = 1e200
    Xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda().t()
    p = pg.pod(Xd, remove_mean=False, energy=0.9, prec=1, check=False)      # binary32 working copy
    assert torch.isnan(p.S).any()
    w = torch.full((900,), 1e300, dtype=torch.float64, device="cuda")
    q = pg.pod(Xd * 1e10, w=w, remove_mean=False, energy=0.9, check=False)
    assert torch.isnan(q.S).any()
    torch.cuda.synchronize()
