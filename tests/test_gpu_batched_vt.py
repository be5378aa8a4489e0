"""Right vectors of batched windows past the kept modes (mixed precision):
orthonormal to binary64 rounding also in a crowd of close singular values, at
a noise floor, in the direction that the removed mean leaves, for rank-
deficient windows, and without any kept mode."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")


def _window(N, M, kind, seed):
    rng = np.random.default_rng(seed)
    Q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    if kind == "crowd":                  # a few structures, then equal values
        s = np.where(np.arange(M) < 4, 2.0 ** -np.arange(M), 1e-2)
    elif kind == "floor":
        s = 2.0 ** -np.arange(M) + 1e-3
    else:                                # rank 5
        s = np.where(np.arange(M) < 5, 2.0 ** -np.arange(M), 0.0)
    Z = np.linalg.qr(rng.standard_normal((N, M)))[0]
    return ((Z * s) @ Q.T).astype(np.float32) + (np.float32(1.0) if kind != "rank" else np.float32(0.0))


@pytest.mark.parametrize("kmodes", [0, 3])
@pytest.mark.parametrize("kind", ["crowd", "floor", "rank"])
def test_right_vectors_are_orthonormal(kind, kmodes):
    sizes = [(400, 16), (900, 33), (1500, 64), (1200, 96), (2000, 128)]
    wins = [_window(N, M, kind, 10 + M) for N, M in sizes]
    b = pg.BatchedPOD([torch.from_numpy(np.ascontiguousarray(X.T)).cuda().t() for X in wins], kmodes=kmodes,
                      prec=pg.PREC_MIXED_3XTF32)
    b.run()
    assert b.status() == pg.OK
    for i, X in enumerate(wins):
        M = X.shape[1]
        VT, S = b.VT[i].cpu().numpy(), b.S[i].cpu().numpy()
        live = np.linalg.norm(VT, axis=1) > 0
        assert live[S > 0].all()
        # Newton-Schulz and Gram-Schmidt in binary64: sums of M products
        assert np.linalg.norm(VT[live] @ VT[live].T - np.eye(live.sum()), 2) <= 4 * M * 2.0 ** -53 * np.sqrt(M)
        Y = X.astype(np.float64) - X.astype(np.float64).mean(1, keepdims=True)
        ref = np.linalg.svd(Y, compute_uv=False)
        assert np.max(np.abs(S - ref)) <= M * 2.0 ** -24 * ref[0]
        # Y v_i has the length of its singular value (M eps_32 S_1)
        assert np.max(np.abs(np.linalg.norm(Y @ VT[live].T, axis=0) - S[live])) <= M * 2.0 ** -24 * ref[0]
