"""Kept modes of small singular values in mixed-precision batches: as accurate
as the Gram matrix's binary64 factor allows, some orders nearer than binary32
leaves bring them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")


@pytest.mark.parametrize("complex_", [True, False])
@pytest.mark.parametrize("N,M", [(3001, 17), (9000, 64), (9001, 127)])
@pytest.mark.parametrize("level", [9e-5, 2e-5, 1.1e-5])
def test_small_kept_modes(level, N, M, complex_):
    rng = np.random.default_rng(M)
    draw = lambda n: rng.standard_normal((n, M)) + (1j * rng.standard_normal((n, M)) if complex_ else 0.0)
    s = np.concatenate([[1.0, 0.5, 0.25, 0.1], level * np.array([3.4, 2.2, 1.5, 1.0]),
                        0.3 * level * 0.99 ** np.arange(M - 8)])
    X = (np.linalg.qr(draw(N))[0] * s) @ np.linalg.qr(draw(M))[0].conj().T
    X = X.astype(np.complex64 if complex_ else np.float32)
    Q, R = np.linalg.qr(X.astype(np.complex128 if complex_ else np.float64))
    u, S, _ = np.linalg.svd(R)
    U = Q @ u[:, :8]
    Xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda().t()
    if complex_:
        b = pg.BatchedSVD([Xd], kmodes=8)
    else:
        b = pg.BatchedPOD([Xd], kmodes=8, prec=pg.PREC_MIXED_3XTF32, remove_mean=False)
    b.run()
    assert b.status() == pg.OK
    modes = b.modes[0].cpu().numpy().astype(U.dtype)
    c = np.sum(U.conj() * modes, axis=0)
    # a binary32 rounding of the modes, and eps_64 / level^2 of squaring over the
    # relative gap of squares between kept modes (0.5): a factor of four on both
    tol = 4 * (2.0 ** -24 + 2.0 ** -53 / level ** 2 / 0.5)
    assert np.max(np.linalg.norm(modes - U * (c / np.abs(c)), axis=0)) <= tol
    assert np.linalg.norm(modes.conj().T @ modes - np.eye(8), 2) <= 2 * tol
    assert np.max(np.abs(b.S[0].cpu().numpy()[:8] - S[:8]) / S[:8]) <= tol
