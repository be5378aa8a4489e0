"""GPU parity of the Gram route of the batched SVDs (mixed precision, default
leaf heights): items at the edges of its tiles (64 and 128 columns, 32-column
Jacobi steps, 128 rows), odd alignments, windows next to bins, and items that
it must hand to the Householder kernel (rank-deficient, equal or zero
singular values among the kept ones), each against the oracle."""
import numpy as np
import pytest

import oracle
import synth
from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")


def _dev(X, dtype=None, shift=0):
    """Column-major CUDA tensor, its first entry `shift` elements into an allocation with ld > rows."""
    X = np.asarray(X)
    N, M = X.shape
    t = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
    t = t if dtype is None else t.to(dtype)
    if not shift:
        return t.t()
    big = torch.zeros((M, N + 2 * shift + 1), dtype=t.dtype, device="cuda")
    big[:, shift:shift + N] = t
    return big[:, shift:shift + N].t()


def _bin(N, Nb, seed, decades=2.0):
    s = 10.0 ** (-decades * np.arange(Nb) / max(Nb - 1, 1))
    return synth.complex_known_spectrum(N, Nb, s=s, seeds=(seed, seed + 1), dtype=np.complex64)[0]


def _check_bin(X, S, U, k):
    U_ref, S_ref, _, _ = oracle.zsvd(X.astype(np.complex128))
    assert np.max(np.abs(S - S_ref)) <= 2e-6 * S_ref[0]
    U = U.astype(np.complex128)
    assert np.linalg.norm(U.conj().T @ U - np.eye(k), 2) <= 1e-5
    for grp in parity.clusters(S_ref):
        grp = [i for i in grp if i < k and S_ref[i] >= 1e-3 * S_ref[0]]
        if not grp:
            continue
        G = U[:, grp].conj().T @ U_ref[:, grp]
        assert np.linalg.svd(G, compute_uv=False).min() >= 1 - 1e-6
        if len(grp) == 1:       # the phase rule too
            assert np.linalg.norm(U[:, grp[0]] - U_ref[:, grp[0]]) <= 2e-3


@pytest.mark.parametrize("kmodes", [0, 4, 32])
def test_bins_at_tile_edges(kmodes):
    sizes = [(1, 1), (5, 2), (64, 31), (127, 32), (129, 33), (500, 63), (513, 64), (300, 65), (1000, 96), (2049, 97),
             (700, 127), (1025, 128)]
    bins = [_bin(N, Nb, 400 + i) for i, (N, Nb) in enumerate(sizes)]
    b = pg.BatchedSVD([_dev(X, shift=i % 3) for i, X in enumerate(bins)], kmodes=kmodes)
    b.run()
    assert b.status() == pg.OK
    S1 = b.S_all.clone()
    for f, X in enumerate(bins):
        _check_bin(X, b.S[f].cpu().numpy(), b.modes[f].cpu().numpy(), b.k[f])
    b.run()
    torch.cuda.synchronize()
    assert torch.equal(S1, b.S_all)


def test_items_left_to_the_householder_kernel():
    rng = np.random.default_rng(7)
    N = 900
    rank3 = (rng.standard_normal((N, 3)) + 1j * rng.standard_normal((N, 3))) @ rng.standard_normal((3, 20))
    steep = _bin(N, 24, 500, decades=6.0)
    equal = synth.unitary_columns(N, 16, 501)
    bins = [rank3.astype(np.complex64), steep, equal.astype(np.complex64), np.zeros((N, 8), np.complex64), _bin(N, 40, 502)]
    b = pg.BatchedSVD([_dev(X) for X in bins], kmodes=8, leaf_rows=None)
    hinted = pg.BatchedSVD([_dev(X) for X in bins], kmodes=8, leaf_rows=[300] * len(bins))
    for x in (b, hinted):
        x.run()
        assert x.status() == pg.OK
    for f, X in enumerate(bins):
        S_ref = oracle.zsvd(X.astype(np.complex128))[1]
        assert np.max(np.abs(b.S[f].cpu().numpy() - S_ref)) <= 2e-6 * max(S_ref[0], 1e-30)
        U = b.modes[f].cpu().numpy().astype(np.complex128)
        assert np.linalg.norm(U.conj().T @ U - np.eye(8), 2) <= 1e-5
        U2 = hinted.modes[f].cpu().numpy().astype(np.complex128)
        assert np.linalg.norm(U2.conj().T @ U2 - np.eye(8), 2) <= 1e-5


@pytest.mark.parametrize("mode_kind", [0, 1])
def test_windows_and_bins(mode_kind):
    shapes = [(40, 1, np.float32), (300, 30, np.float64), (1000, 64, np.float32), (777, 65, np.float32),
              (1300, 128, np.float64), (9, 9, np.float32)]
    wins, ws = [], []
    for i, (N, M, ft) in enumerate(shapes):
        rng = np.random.default_rng(600 + i)
        s = 2.0 ** -np.arange(M)
        X = (rng.standard_normal((N, M)) * (s + 1e-3)) @ np.linalg.qr(rng.standard_normal((M, M)))[0] + 1.0
        wins.append(np.asfortranarray(X.astype(ft)))
        ws.append(synth.log_uniform_weights(N, seed=i) if i % 2 else None)
    bins = [_bin(800, 50, 610)]
    bp = pg.BatchedPOD([_dev(X) for X in wins], weights=[None if w is None else torch.from_numpy(w).cuda() for w in ws],
                       mode_kind=mode_kind, kmodes=5, prec=pg.PREC_MIXED_3XTF32, bins=[_dev(X) for X in bins])
    bp.run()
    assert bp.status() == pg.OK
    for i, (X, w) in enumerate(zip(wins, ws)):
        if X.shape[1] == 1:
            continue               # its mean is itself: a zero matrix
        ref = oracle.pod(X.astype(np.float64), w=w, remove_mean=True, mode_kind=mode_kind)
        S = bp.S[i].cpu().numpy()
        assert np.max(np.abs(S - ref["S"])) <= 2e-6 * ref["S"][0], i
        keep = [j for j in range(bp.k[i]) if ref["S"][j] >= 1e-3 * ref["S"][0]]
        wt = w if mode_kind else None
        parity.check_vectors(bp.modes[i].cpu().numpy().astype(np.float64)[:, keep], ref["U"][:, keep], ref["S"][keep],
                             ncols=len(keep), weight=wt)
        parity.check_vectors(bp.VT[i].cpu().numpy().T[:, keep], ref["VT"].T[:, keep], ref["S"][keep], ncols=len(keep))
        np.testing.assert_allclose(bp.mean[i].cpu().numpy(), ref["mean"], rtol=0, atol=1e-13)
    _check_bin(bins[0], bp.S[-1].cpu().numpy(), bp.modes[-1].cpu().numpy(), bp.k[-1])
    X = wins[1].copy()
    X[3, 4] = np.inf
    bad = pg.BatchedPOD([_dev(X)], kmodes=2, prec=pg.PREC_MIXED_3XTF32)
    bad.run()
    assert bad.status() == pg.ERR_NONFINITE
