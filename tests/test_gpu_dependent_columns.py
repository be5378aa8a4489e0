"""Snapshots that depend on earlier ones (a zero first snapshot, one written
twice, a run of nearly parallel ones) before independent ones, in calls that
the device takes from the Gram route to the Householder route: the Cholesky
factor and the Householder R of such a matrix differ by more than row signs.
Modes against LAPACK column by column, the adjoint against the one of an
explicit leaf height."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")

KINDS = ["zero", "repeated", "parallel"]


def _field(N, M, kind, seed, s):
    """N x M with singular values near s (M - 1 of them) and dependent first columns."""
    rng = np.random.default_rng(seed)
    Q = np.linalg.qr(rng.standard_normal((N, M - 1)))[0]
    B = (Q * s) @ synth.haar_orthogonal(M - 1, seed + 1).T
    if kind == "zero":
        X = np.concatenate([np.zeros((N, 1)), B], axis=1)
    elif kind == "repeated":
        X = np.concatenate([B[:, :1], B], axis=1)
    else:
        X = np.concatenate([B[:, :1], B], axis=1)
        for j in range(1, 10):
            X[:, j] = X[:, 0] * (1 + 0.01 * j) + 1e-7 * np.linalg.norm(X[:, 0]) / np.sqrt(N) * rng.standard_normal(N)
    return np.asfortranarray(X)


def _dev(X, dtype):
    return torch.from_numpy(np.ascontiguousarray(X.T)).to("cuda").to(dtype).t()


def _reference(X):
    U, S, VT = np.linalg.svd(X, full_matrices=False)
    sg = np.sign(VT[np.arange(len(S)), np.argmax(np.abs(VT), axis=1)])
    return U * sg, S, VT * sg[:, None]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("N,M", [(4096, 24), (9000, 270)])
def test_modes_after_the_fallback(N, M, kind, prec):
    # a decaying part down to 1e-2, then a tail that no direct product can hold
    k = M // 3
    s = np.concatenate([10.0 ** (-2.0 * np.arange(k) / k), 1e-7 * 10.0 ** (-1.0 * np.arange(M - 1 - k) / M)])
    X = _field(N, M, kind, 5 + M, s)
    Xd = _dev(X, torch.float32 if prec else torch.float64)
    X = Xd.double().cpu().numpy()
    p = pg.pod(Xd, remove_mean=False, r_max=M - 1, prec=prec)
    U, S, VT = _reference(X)
    eps = 2.0 ** -24 if prec else 2.0 ** -53
    # a backward error of M eps S_1 in Y moves a singular value by as much and
    # a vector by that over the gap to the next value
    back = M * eps * S[0]
    Ug, Sg, Vg = p.U.double().cpu().numpy(), p.S.cpu().numpy(), p.VT.cpu().numpy()
    assert np.max(np.abs(Sg - S)) <= back
    gap = np.minimum(np.abs(np.diff(S, prepend=np.inf)), np.abs(np.diff(S, append=-np.inf)))
    n = k - 1                                       # well above the tail
    assert np.all(np.linalg.norm(X @ Vg[:n].T - Ug[:, :n] * Sg[:n], axis=0) <= back)
    for i in range(n):
        assert np.linalg.norm(Ug[:, i] - U[:, i]) <= back / gap[i], i
    assert np.linalg.norm(Ug.T @ Ug - np.eye(M - 1), 2) <= M * eps


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("N,M", [(4096, 24), (6000, 150)])
def test_adjoint_after_the_fallback(N, M, kind, prec):
    """A cotangent on a small singular value sends the adjoint of a Gram
    forward to a factorisation of its own."""
    s = np.concatenate([2.0 ** -np.arange(8.0), 1e-6 * 0.9 ** np.arange(M - 9)])
    X = _dev(_field(N, M, kind, 7 + M, s), torch.float32 if prec else torch.float64)
    g = torch.Generator(device="cuda")
    out = []
    for b in (0, 1000):
        f = pg.pod(X, remove_mean=False, energy=0.999, prec=prec, leaf_rows=b)
        dU = torch.randn((f.r, N), dtype=torch.float64, device="cuda", generator=g.manual_seed(1)).t() / N ** 0.5
        dS = torch.randn(M, dtype=torch.float64, device="cuda", generator=g.manual_seed(2))
        dS[f.r:] = 0.0
        dS[10] = 1e-6
        out.append(pg.pod_backward(f, (N, M), None, False, 0, b, M, dU=dU, dS=dS))
    # kept values are at least a factor of two apart (1/16 of the largest or
    # more), so the cotangent moves by at most some 1e2 M eps; u_10 itself,
    # uncertain in binary32, enters with 1e-6
    eps = 2.0 ** -24 if prec else 2.0 ** -53
    tol = 1e2 * M * eps + (1e-6 if prec else 1e-6 * M * eps / 1e-7)
    assert torch.norm(out[0] - out[1]) <= tol * torch.norm(out[1])
