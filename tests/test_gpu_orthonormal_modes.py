"""Modes of the Gram route in binary64 are as orthonormal as the small SVD leaves
its vectors, whatever the smallest kept value (Y V S^-1 alone: to eps s_1 / s_r)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")


@pytest.mark.parametrize("ratio", [2.0, 15.0, 17.0, 1e3, 9e3])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("N,M,r", [(900, 9, 8), (3001, 40, 7), (4000, 129, 65), (5000, 260, 33)])
def test_modes_are_orthonormal(N, M, r, weighted, ratio):
    rng = np.random.default_rng(N)
    s = ratio ** (-np.arange(M) / (r - 1.0))
    s[r:] = s[r - 1] * 0.5
    X = (np.linalg.qr(rng.standard_normal((N, M)))[0] * s) @ synth.haar_orthogonal(M, 4).T
    w = synth.log_uniform_weights(N, seed=3) if weighted else None
    if weighted:
        X /= np.sqrt(w)[:, None]
    Xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda().t()
    p = pg.pod(Xd, w=None if w is None else torch.from_numpy(w).cuda(), remove_mean=False, r_max=r,
               mode_kind=int(weighted))
    U = p.U.cpu().numpy()
    if weighted:
        U = U * np.sqrt(w)[:, None]
    # the small SVD stops at cosines of M eps between right vectors' images, for
    # each of r modes; nothing may grow with s_1 / s_r on top of that
    assert np.linalg.norm(U.T @ U - np.eye(r), 2) <= r * M * 2.0 ** -53
    Y = X if w is None else X * np.sqrt(w)[:, None]
    # they still are left vectors: |Y v - s u| within the same of S_1
    V, S = p.VT.cpu().numpy()[:r].T, p.S.cpu().numpy()[:r]
    assert np.max(np.linalg.norm(Y @ V - U * S, axis=0)) <= r * M * 2.0 ** -53 * S[0]
