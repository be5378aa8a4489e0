"""GPU parity of the preconditioned small SVD (binary32 block Jacobi, binary64
simultaneous rotations, then the binary64 sweeps if any pair is left) at the
edges of its blocks (16 and 32 columns, cluster and grid launches) and on the
spectra that decide its path: graded, clustered at a floor, double singular
values, rank deficient, and scales far from one."""
import numpy as np
import pytest

from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")


def _r(M, kind, seed):
    rng = np.random.default_rng(seed)
    Q1 = np.linalg.qr(rng.standard_normal((2 * M, M)))[0]
    Q2 = np.linalg.qr(rng.standard_normal((M, M)))[0]
    i = np.arange(M)
    s = {"graded": 10.0 ** (-8.0 * i / max(M - 1, 1)), "floor": 10.0 ** (-6.0 * i / 255) + 1e-5,
         "double": 2.0 ** -(i // 2).astype(float) + 1e-4, "equal": np.ones(M),
         "deficient": np.where(i < (M + 1) // 2, 1.0 / (1 + i), 0.0), "huge": 1e60 * 10.0 ** (-3.0 * i / M),
         "tiny": 1e-60 * 10.0 ** (-3.0 * i / M)}[kind]
    return np.asfortranarray(np.linalg.qr((Q1 * s) @ Q2.T)[1])


@pytest.mark.parametrize("M", [11, 12, 16, 17, 32, 33, 64, 65, 129, 256, 272, 273])
@pytest.mark.parametrize("kind", ["graded", "floor", "double", "equal", "deficient", "huge", "tiny"])
def test_preconditioned_svd(M, kind):
    R = _r(M, kind, M)
    U, S, VT, sweeps = pg.svd_small(torch.from_numpy(np.ascontiguousarray(R.T)).cuda().t())
    U, S, V = U.cpu().numpy(), S.cpu().numpy(), VT.cpu().numpy().T
    S_ref = np.linalg.svd(R / S[0], compute_uv=False) * S[0]
    parity.check_sigma(S / S[0], S_ref / S[0])
    # the bounds of the small SVD's own tests: rounding grows with the rotations
    assert np.linalg.norm(R / S[0] - (U * (S / S[0])) @ V.T) <= max(1e-13, 1e-15 * M) * np.linalg.norm(R / S[0])
    assert np.linalg.norm(U.T @ U - np.eye(M), 2) <= max(1e-13, 5e-15 * M)
    keep = S > 1e-14 * M * S[0]      # right vectors of rounding-level values are rounding
    Vk = V[:, keep]
    assert np.linalg.norm(Vk.T @ Vk - np.eye(Vk.shape[1]), 2) <= max(1e-13, 5e-15 * M)
    assert 1 <= sweeps <= 60


def test_preconditioned_svd_zero_and_nan():
    M = 40
    U, S, VT, _ = pg.svd_small(torch.zeros((M, M), dtype=torch.float64, device="cuda"))
    assert torch.all(S == 0)
    for Q in (U, VT):
        assert torch.linalg.norm(Q.t() @ Q - torch.eye(M, dtype=torch.float64, device="cuda")) < 1e-13
    R = torch.eye(M, dtype=torch.float64, device="cuda")
    R[3, 5] = float("nan")
    pg.svd_small(R, check=False)     # ends, whatever its outputs
    torch.cuda.synchronize()
