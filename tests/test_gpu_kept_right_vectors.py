"""Kept right vectors of batched windows (mixed precision) beside a crowd of
close values: as accurate as their own columns were diagonalised, whatever the
crowd's vectors need to become orthonormal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")


@pytest.mark.parametrize("seed", range(3))
@pytest.mark.parametrize("N,M", [(1500, 33), (3000, 64), (4000, 96), (5000, 128)])
def test_kept_rows(N, M, seed):
    rng = np.random.default_rng(100 * M + seed)
    s = np.where(np.arange(M) < 3, 2.0 ** -np.arange(M), 1e-2)
    X = (np.linalg.qr(rng.standard_normal((N, M)))[0] * s) @ np.linalg.qr(rng.standard_normal((M, M)))[0].T
    X = X.astype(np.float32)
    b = pg.BatchedPOD([torch.from_numpy(np.ascontiguousarray(X.T)).cuda().t()], kmodes=3, prec=pg.PREC_MIXED_3XTF32,
                      remove_mean=False)
    b.run()
    assert b.status() == pg.OK
    V = np.linalg.svd(X.astype(np.float64), full_matrices=False)[2][:3]
    VT = b.VT[0].cpu().numpy()[:3]
    VT = VT * np.sign(np.sum(V * VT, axis=1))[:, None]
    # cosines of at most 1e-6 with the crowd turn a kept vector by that times the
    # ratio of the values (4e-2 at most)
    assert np.max(np.linalg.norm(VT - V, axis=1)) <= 5e-8
