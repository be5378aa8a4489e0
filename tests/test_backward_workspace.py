"""The adjoint's workspace: room for a factorisation of Y lies in the region of
dY, so the automatic leaf height needs little more than an explicit one (CPU);
and the adjoint that uses it that way, a few columns of dY at a time (GPU)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")

pg = pytest.importorskip("paper_2405_15529_gb300")


@pytest.mark.parametrize("N,M,r,prec", [(1 << 22, 256, 43, 0), (1 << 22, 256, 43, 1), (1 << 20, 128, 128, 0),
                                        (300001, 700, 128, 1), (262144, 64, 20, 0)])
def test_automatic_height_needs_little_more(N, M, r, prec):
    from paper_2405_15529_gb300 import _build
    _build.build()
    lib = pg.load_library()
    P = pg.leaf_count(N, M, 0)
    auto = lib.pylom_pod_backward_workspace_size(N, M, 0, r, prec)
    if prec:
        P = min(P, 152)
    one = lib.pylom_pod_backward_workspace_size(N, M, N // P, r, prec)
    # 16 columns of dY, the reflectors' small factors and R slots, some M x M matrices
    assert one < auto <= one + 16 * 8 * N + (4 * P + 40) * 8 * M * M + 64 * N


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dx_dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("N,M,weighted,mean", [(2003, 12, False, True), (4001, 40, True, True), (3000, 33, True, False)])
def test_adjoint_beside_its_reflectors(N, M, weighted, mean, dx_dtype, prec):
    """A cotangent on a small singular value: Y is factored in the region of dY."""
    s = np.concatenate([2.0 ** -np.arange(6.0), 1e-6 * 0.8 ** np.arange(M - 6)])
    rng = np.random.default_rng(M)
    X = (np.linalg.qr(rng.standard_normal((N, M)))[0] * s) @ synth.haar_orthogonal(M, 3).T
    w = synth.log_uniform_weights(N, seed=2, lo=0.1) if weighted else None
    if mean:
        X = X + 0.01 * rng.standard_normal((N, 1))
    Xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda().to(torch.float32 if prec else torch.float64).t()
    wd = None if w is None else torch.from_numpy(w).cuda()
    g = torch.Generator(device="cuda")
    out = []
    for b in (0, 1000):
        f = pg.pod(Xd, w=wd, remove_mean=mean, r_max=3, mode_kind=int(weighted), prec=prec, leaf_rows=b)
        dU = torch.randn((f.r, N), dtype=torch.float64, device="cuda", generator=g.manual_seed(1)).t() / N ** 0.5
        dS = torch.randn(M, dtype=torch.float64, device="cuda", generator=g.manual_seed(2))
        dS[3:] = 0.0
        dS[7] = 1e-6
        out.append(pg.pod_backward(f, (N, M), wd, mean, int(weighted), b, 3, dU=dU, dS=dS, dx_dtype=dx_dtype).double())
    eps = 2.0 ** -24 if prec or dx_dtype == torch.float32 else 2.0 ** -53
    # kept values a factor of two apart, 1/4 of the largest or more: some 1e2 M eps;
    # u_7 itself, uncertain in binary32, enters with 1e-6
    tol = 1e2 * M * eps + (1e-6 if prec else 1e-6 * M * 2.0 ** -53 / 1e-7)
    assert torch.norm(out[0] - out[1]) <= tol * torch.norm(out[1])
    if mean:
        assert torch.max(torch.abs(out[0].sum(1))) <= 1e2 * M * eps * torch.norm(out[0])
