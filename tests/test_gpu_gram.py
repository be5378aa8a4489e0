"""GPU parity of the Gram route of the POD and the DMD (exact integer Gram
matrix on the tensor cores, double-double Cholesky factor, direct modes
product), which calls with the automatic leaf height and an energy share
take, against the FP64 oracle and against the Householder route that an
explicit leaf height takes -- at the edges of its tiles (128 rows, 64 and
128 columns, 32-column stages), over layouts, types, weights and spectra,
and through the adjoint, which then factors the forward's Y itself."""
import numpy as np
import pytest

import oracle
import synth
from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")


def _dev(X, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(np.asarray(X).T)).to("cuda")
    return (t if dtype is None else t.to(dtype)).t()


def _field(N, M, seed, decades=3.0):
    """Well separated singular values over `decades`, on a mean field."""
    rng = np.random.default_rng(seed)
    Q2 = synth.haar_orthogonal(M, seed + 1) if M > 1 else np.ones((1, 1))
    s = synth.spectrum(M, decades=decades)
    X = (rng.standard_normal((N, M)) * s[None, :]) @ Q2.T
    X += (1.0 + 0.5 * np.cos(2.0 * np.pi * np.arange(N) / N))[:, None]
    return np.asfortranarray(X)


# rows and columns around the tile edges
SHAPES = [(129, 1), (128, 2), (127, 31), (257, 33), (1000, 63), (640, 64), (1025, 65), (2049, 127), (2048, 128),
          (3001, 129), (1537, 192), (4099, 257)]


@pytest.mark.parametrize("mode_kind,weighted,mean", [(0, False, False), (1, True, True)])
@pytest.mark.parametrize("N,M", SHAPES)
def test_gram_pod_matches_oracle(N, M, weighted, mean, mode_kind):
    mean = mean and M > 1
    X = _field(N, M, N + M)
    w = synth.log_uniform_weights(N, seed=M) if weighted else None
    ref = oracle.pod(X, w=w, remove_mean=mean, energy=0.999, mode_kind=mode_kind)
    res = pg.pod(_dev(X), w=None if w is None else torch.from_numpy(w).cuda(), remove_mean=mean, energy=0.999,
                 mode_kind=mode_kind)
    parity.check_sigma(res.S.cpu().numpy(), ref["S"])
    assert res.r == ref["r"]
    wt = w if mode_kind == 1 else None
    U = res.U.cpu().numpy()
    parity.check_vectors(U, ref["U"], ref["S"], ncols=res.r, weight=wt)
    parity.check_vectors(res.VT.cpu().numpy().T, ref["VT"].T, ref["S"], ncols=res.r)
    np.testing.assert_allclose(res.mean.cpu().numpy(), ref["mean"], rtol=0, atol=1e-14 * np.abs(X).max())
    # u_k = Y v_k / s_k: the roundings of the r right vectors (a few M eps
    # each from the Jacobi rotations) grow by at most s_1 / s_r
    kappa = ref["S"][0] / ref["S"][res.r - 1]
    assert parity.orthonormality(U, weight=wt) <= res.r * 4 * max(M, 16) * 2.0 ** -53 * kappa


@pytest.mark.parametrize("prec,dtype", [(0, torch.float64), (0, torch.float32), (1, torch.float32),
                                        (1, torch.float64)])
@pytest.mark.parametrize("layout", ["columns", "rows", "slice", "shifted"])
def test_gram_pod_agrees_with_householder_route(prec, dtype, layout):
    N, M = 5003, 70
    X = _dev(_field(N, M, 11), dtype)
    big = torch.zeros((M, N + 6), dtype=dtype, device="cuda")
    if layout == "rows":
        X = X.contiguous()
    elif layout == "slice":            # ld > N
        big[:, :N] = X.t()
        X = big[:, :N].t()
    elif layout == "shifted":          # columns that start off a 16-byte boundary
        big[:, 3:N + 3] = X.t()
        X = big[:, 3:N + 3].t()
    w = torch.from_numpy(synth.log_uniform_weights(N, seed=5)).cuda()
    a = pg.pod(X, w=w, energy=0.99, prec=prec)
    b = pg.pod(X, w=w, energy=0.99, prec=prec, leaf_rows=1000)
    assert a.r == b.r
    S = b.S.cpu().numpy()
    # the mixed routes round differently: each is within 2e-6 S_max of exact
    tol = 4e-6 if prec else 2e-12
    assert np.max(np.abs(a.S.cpu().numpy() - S)) <= tol * S[0]
    parity.check_vectors(a.U.double().cpu().numpy(), b.U.double().cpu().numpy(), S, ncols=a.r)
    assert torch.allclose(a.mean, b.mean, rtol=0, atol=1e-14)
    c = pg.pod(X, w=w, energy=0.99, prec=prec)
    assert torch.equal(a.S, c.S) and torch.equal(a.U, c.U) and torch.equal(a.VT, c.VT)


@pytest.mark.parametrize("prec", [0, 1])
def test_gram_pod_extreme_columns(prec):
    """Columns of very different scale, a zero column, equal columns, and
    columns whose largest entry is far above the rest."""
    N, M = 4000, 40
    rng = np.random.default_rng(3)
    X = rng.standard_normal((N, M))
    X[:, 1] = 0.0
    X[:, 3] = X[:, 2]
    X[:, 4] *= 1e-12
    X[:, 5] *= 1e12 if prec == 0 else 1e3
    X[17, 6] = 3e3
    X = np.asfortranarray(X.astype(np.float32 if prec else np.float64))
    ref = oracle.pod(X.astype(np.float64), remove_mean=False, energy=0.9)
    res = pg.pod(_dev(X), remove_mean=False, energy=0.9, prec=prec)
    S = res.S.cpu().numpy()
    assert res.r == ref["r"]
    assert np.max(np.abs(S - ref["S"])) <= (2e-6 if prec else 1e-12) * ref["S"][0]
    parity.check_vectors(res.U.double().cpu().numpy(), ref["U"], ref["S"], ncols=res.r)


def test_gram_pod_zero_matrix_and_nonfinite():
    X = np.repeat(np.round(100 * np.random.default_rng(4).standard_normal((300, 1))), 12, axis=1)
    X = np.asfortranarray(X)
    res = pg.pod(_dev(X), remove_mean=True, energy=0.9)
    assert torch.all(res.S == 0.0) and res.r == 12
    assert parity.orthonormality(res.U.cpu().numpy()) < 1e-13
    for bad in (np.nan, np.inf):
        Y = _field(1000, 10, 1)
        Y[17, 3] = bad
        for prec in (0, 1):
            with pytest.raises(pg.PylomError) as ei:
                pg.pod(_dev(Y), energy=0.9, prec=prec)
            assert ei.value.status == pg.ERR_NONFINITE
    w = torch.ones(1000, dtype=torch.float64, device="cuda")
    w[999] = -1.0
    with pytest.raises(pg.PylomError) as ei:
        pg.pod(_dev(_field(1000, 10, 1)), w=w, energy=0.9)
    assert ei.value.status == pg.ERR_NONFINITE


@pytest.mark.parametrize("prec", [0, 1])
def test_adjoint_of_a_gram_forward(prec):
    """pod_backward after a forward that left Y unfactored equals the one
    after a forward with reflectors (same r)."""
    N, M = 6000, 40
    X = _dev(_field(N, M, 21, decades=1.0), torch.float32 if prec else torch.float64)
    a = pg.pod(X, energy=0.9, prec=prec)
    b = pg.pod(X, energy=0.9, prec=prec, leaf_rows=1500)
    assert a.r == b.r
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    dU = torch.randn((a.r, N), dtype=torch.float64, device="cuda", generator=g).t()
    dS = torch.randn(M, dtype=torch.float64, device="cuda", generator=g)
    ga = pg.pod_backward(a, (N, M), None, True, 0, 0, M, dU=dU, dS=dS)
    gb = pg.pod_backward(b, (N, M), None, True, 0, 1500, M, dU=dU, dS=dS)
    again = pg.pod_backward(a, (N, M), None, True, 0, 0, M, dU=dU, dS=dS)
    # couplings 1 / (s_j^2 - s_i^2) of a one-decade spectrum amplify the
    # forwards' roundings (1e-14, 1e-7) by about 1e3
    assert torch.norm(ga - gb) <= (1e-3 if prec else 1e-10) * torch.norm(gb)
    assert torch.equal(ga, again)


def test_gram_dmd_agrees_with_householder_route():
    N, M, K = 5001, 50, 8
    lam, amp = synth.oscillation_params(K, seed=3)
    D, _ = synth.oscillations(N, M, lam, amp, seed=4, noise=1e-6, offset=0.5)
    a = pg.dmd(_dev(D), r_max=2 * K)
    b = pg.dmd(_dev(D), r_max=2 * K, leaf_rows=1000)
    assert a.r == b.r
    # perturbations of 1e-14 over the smallest kept singular value (1e-2 of the largest)
    assert torch.max(torch.abs(a.mu - b.mu)) <= 1e-11
    assert torch.norm(a.b - b.b) <= 1e-10 * torch.norm(b.b)
    assert torch.norm(a.Phi_packed - b.Phi_packed) <= 1e-10 * torch.norm(b.Phi_packed)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kind", ["decay", "deficient", "steep", "zero"])
@pytest.mark.parametrize("N,M,r", [(3001, 40, 12), (70000, 65, 30)])
def test_rank_limited_pod(N, M, r, kind, prec):
    """r_max < M without an energy share: the device decides between the
    direct product and the Householder route (values too small among the
    kept ones); modes are orthonormal either way."""
    rng = np.random.default_rng(N)
    if kind == "decay":
        X = _field(N, M, 31, decades=2.0)
    elif kind == "deficient":             # rank 5 < r
        X = rng.standard_normal((N, 5)) @ rng.standard_normal((5, M))
    elif kind == "steep":
        X = _field(N, M, 33, decades=14.0)
    else:
        X = np.ones((N, M))
    X = np.asfortranarray(X.astype(np.float32 if prec else np.float64))
    Xd = _dev(X)
    a = pg.pod(Xd, r_max=r, prec=prec)
    b = pg.pod(Xd, r_max=r, prec=prec, leaf_rows=1000)
    assert a.r == b.r == r
    S = b.S.cpu().numpy()
    assert np.max(np.abs(a.S.cpu().numpy() - S)) <= (4e-6 if prec else 2e-12) * max(S[0], 1e-300)
    U = a.U.double().cpu().numpy()
    assert parity.orthonormality(U) <= (1e-5 if prec else 1e-11 if kind == "decay" else 1e-12 * r)
    keep = [i for i in range(r) if S[i] >= (1e-3 if prec else 1e-8) * S[0] > 0]
    if keep:
        parity.check_vectors(U[:, keep], b.U.double().cpu().numpy()[:, keep], S[keep], ncols=len(keep))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kind", ["decay", "steep"])
@pytest.mark.parametrize("mode_kind,weighted,mean", [(0, False, True), (1, True, False)])
@pytest.mark.parametrize("N,M,r", [(2500, 33, 6), (5000, 130, 20)])
def test_adjoint_after_rank_limited_pod(N, M, r, mode_kind, weighted, mean, kind, prec):
    if kind == "steep" and (prec or weighted):
        pytest.skip("one steep case: the forward leaves it to the Householder route")
    X = _field(N, M, 41, decades=1.0 if kind == "decay" else 1.2 * (M - 1))   # steep: s_r = 1e-6 s_1 and less
    dt = torch.float32 if prec else torch.float64
    Xd = _dev(X, dt)
    w = torch.from_numpy(synth.log_uniform_weights(N, seed=6, lo=0.1)).cuda() if weighted else None
    g = torch.Generator(device="cuda")
    full = kind == "decay" and not mean      # cotangents of all values and right vectors
    out = []
    for b in (0, 700):
        f = pg.pod(Xd, w=w, remove_mean=mean, r_max=r, mode_kind=mode_kind, prec=prec, leaf_rows=b)
        dU = torch.randn((f.r, N), dtype=torch.float64, device="cuda", generator=g.manual_seed(3)).t()
        dS = torch.randn(M, dtype=torch.float64, device="cuda", generator=g.manual_seed(4))
        dVT = torch.randn((M, M), dtype=torch.float64, device="cuda", generator=g.manual_seed(5))
        if kind == "steep":
            dU[:, 3:] = 0.0
        if not full:
            dS[3 if kind == "steep" else r:] = 0.0
        out.append(pg.pod_backward(f, (N, M), w, mean, mode_kind, b, r, dU=dU, dS=dS, dVT=dVT if full else None))
    # couplings 1 / (s_j^2 - s_i^2) of the closest values (2 % apart for M =
    # 130) amplify the forwards' roundings; 1e-3 between the steep ones
    assert torch.norm(out[0] - out[1]) <= (2e-3 if prec else 1e-9) * torch.norm(out[1])
