"""Jacobi iterations on matrices with exactly zero singular values that no row
of the factor shows (a zero first snapshot, zero rows): they end, with the
singular values and vectors of LAPACK, through every entry that iterates."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")


@pytest.mark.parametrize("M", [5, 11, 24, 65, 270])
@pytest.mark.parametrize("zeros", [1, 3])
@pytest.mark.parametrize("scale", [1.0, 1e90, 1e-90])
def test_small_svd_with_zero_columns(M, zeros, scale):
    rng = np.random.default_rng(M)
    R = rng.standard_normal((M, M)) * scale
    R[:, :zeros] = 0.0
    U, S, VT, _ = pg.svd_small(torch.from_numpy(np.ascontiguousarray(R.T)).cuda().t())
    U, S, VT = U.cpu().numpy(), S.cpu().numpy(), VT.cpu().numpy()
    S_ref = np.linalg.svd(R / scale, compute_uv=False)
    # backward stable: each value within M eps S_1 (rotations round a few times M)
    assert np.max(np.abs(S / scale - S_ref)) <= 8 * M * 2.0 ** -53 * S_ref[0]
    assert np.linalg.norm(R / scale - (U * (S / scale)) @ VT) <= 8 * M * 2.0 ** -53 * np.linalg.norm(S_ref)
    for Q in (U.T, VT[:M - zeros]):
        assert np.linalg.norm(Q @ Q.T - np.eye(len(Q)), 2) <= 8 * M * 2.0 ** -53


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("leaf_rows", [0, 512])
def test_pod_with_a_zero_first_snapshot(leaf_rows, prec):
    rng = np.random.default_rng(2)
    X = rng.standard_normal((2000, 30))
    X[:, 0] = 0.0
    Xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda().t()
    p = pg.pod(Xd.float() if prec else Xd, remove_mean=False, leaf_rows=leaf_rows, prec=prec)
    S = np.linalg.svd(X, compute_uv=False)
    eps = 2.0 ** -24 if prec else 2.0 ** -53
    assert np.max(np.abs(p.S.cpu().numpy() - S)) <= 30 * eps * S[0]
    U = p.U.double().cpu().numpy()
    assert np.linalg.norm(U.T @ U - np.eye(30), 2) <= 60 * eps


@pytest.mark.parametrize("prec", [0, 1])
def test_batched_bins_with_a_zero_first_column(prec):
    g = torch.Generator(device="cuda").manual_seed(3)
    Q = torch.randn((20, 900), dtype=torch.complex64, device="cuda", generator=g).t()
    Q[:, 0] = 0
    b = pg.BatchedSVD([Q], kmodes=4, prec=prec, leaf_rows=[300])
    b.run()
    assert b.status() == pg.OK
    assert b.S_all[-1] <= 20 * (2.0 ** -24 if prec else 2.0 ** -53) * b.S_all[0]
