"""Right vectors of exactly zero singular values whose directions are spread
evenly over all snapshots, as the one that the removed mean leaves: unit length
and orthogonal to the others."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")


def _orthonormal(VT):
    M = len(VT)
    # each pair of rows to the cosine at which the iteration stops, M eps
    return np.max(np.abs(VT @ VT.T - np.eye(M))) <= 4 * M * 2.0 ** -53


@pytest.mark.parametrize("M", [2, 5, 11, 16, 65, 130, 700])
@pytest.mark.parametrize("groups", [1, 2])
def test_even_null_vectors(M, groups):
    """R x = 0 for x constant over each of `groups` ranges of columns."""
    rng = np.random.default_rng(M)
    R = np.zeros((M, M))
    ends = np.linspace(0, M, groups + 1).astype(int)
    T = rng.standard_normal((M - groups, M - groups)) + 3 * np.eye(M - groups)
    c = 0
    for a, b in zip(ends[:-1], ends[1:]):
        n = b - a - 1
        R[:M - groups, a:b - 1] = T[:, c:c + n]
        R[:M - groups, b - 1] = -T[:, c:c + n].sum(1)
        c += n
    U, S, VT, _ = pg.svd_small(torch.from_numpy(np.ascontiguousarray(R.T)).cuda().t())
    U, S, VT = U.cpu().numpy(), S.cpu().numpy(), VT.cpu().numpy()
    assert np.all(S[M - groups:] <= M * 2.0 ** -53 * max(S[0], 1e-300)) and _orthonormal(VT) and _orthonormal(U.T)
    assert np.linalg.norm(R - (U * S) @ VT) <= 8 * M * 2.0 ** -53 * np.linalg.norm(S)


@pytest.mark.parametrize("N,M", [(2000, 16), (5000, 64), (3000, 200)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_pod_without_its_mean(N, M, dtype):
    g = torch.Generator(device="cuda").manual_seed(M)
    X = torch.randn((M, N), dtype=dtype, device="cuda", generator=g).t()
    p = pg.pod(X, remove_mean=True, r_max=M // 3)
    assert _orthonormal(p.VT.cpu().numpy())
    # the null direction of centred snapshots
    assert abs(abs(p.VT[M - 1].sum().item()) - M ** 0.5) <= 1e-9
