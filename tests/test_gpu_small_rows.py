"""Points whose values are small beside the rest of the field (a quiet far
field, variables of different size in one X, cells of very different volume):
their rows of the modes, of the DMD modes and of the adjoint are as accurate,
relative to the row, as those of large rows."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")


def _dev(X, dtype=torch.float64):
    return torch.from_numpy(np.ascontiguousarray(X.T)).to("cuda").to(dtype).t()


def _field(N, M, seed, small, dtype=np.float64, zero_column=False):
    """Decaying spectrum (one decade over M); every third row times `small`,
    one in 40 zero."""
    rng = np.random.default_rng(seed)
    s = 10.0 ** (-np.arange(M) / M)
    X = (rng.standard_normal((N, M)) * s) @ synth.haar_orthogonal(M, seed + 1).T
    X[1::3] *= small
    X[::40] = 0.0
    if zero_column:
        X[:, M // 2] = 0.0
    return np.asfortranarray(X.astype(dtype).astype(np.float64))


def _modes(Y, k):
    U, S, VT = np.linalg.svd(Y, full_matrices=False)
    sg = np.sign(VT[np.arange(len(S)), np.argmax(np.abs(VT), axis=1)])
    V = (VT * sg[:, None]).T
    gap = np.minimum(np.abs(np.diff(S, prepend=np.inf)), np.abs(np.diff(S, append=-np.inf)))
    return (Y @ V[:, :k]) / S[:k], S, gap


def _rows_agree(U, Y, eps, k, scale=1.0):
    """Every row of U against Y v / s: v moves by M eps S_1 / gap, and a row by
    that times its own norm."""
    ref, S, gap = _modes(Y, k)
    rho = np.linalg.norm(Y, axis=1)
    live = rho > 0
    for i in range(k):
        err = np.abs(U[:, i] - ref[:, i] * scale)[live] / (rho[live] / S[i] * (scale[live] if np.ndim(scale) else 1.0))
        assert err.max() <= Y.shape[1] * eps * S[0] / gap[i], (i, err.max())
    assert np.all(U[~live] == 0.0)


@pytest.mark.parametrize("energy,r_max", [(0.9, None), (0.0, 5)])
@pytest.mark.parametrize("zero_column", [False, True])
@pytest.mark.parametrize("small", [0.05, 1e-4, 1e-8, 1e-12, 1e-40])
@pytest.mark.parametrize("N,M", [(1500, 12), (4099, 63), (2100, 130), (3000, 300)])
def test_rows_of_binary64_modes(N, M, small, zero_column, energy, r_max):
    X = _field(N, M, N, small, zero_column=zero_column)
    p = pg.pod(_dev(X), remove_mean=False, energy=energy, r_max=r_max)
    _rows_agree(p.U.cpu().numpy(), X, 2.0 ** -53, 3)


@pytest.mark.parametrize("zero_column", [False, True])
@pytest.mark.parametrize("small", [0.05, 1e-3, 1e-5, 1e-8, 1e-30])
@pytest.mark.parametrize("N,M", [(1500, 12), (4099, 63), (2100, 130), (3000, 300)])
def test_rows_of_mixed_modes(N, M, small, zero_column):
    X = _field(N, M, N, small, np.float32, zero_column)
    p = pg.pod(_dev(X, torch.float32), remove_mean=False, energy=0.9, prec=1)
    _rows_agree(p.U.double().cpu().numpy(), X, 2.0 ** -24, 3)


@pytest.mark.parametrize("prec", [0, 1])
def test_physical_modes_over_uneven_cells(prec):
    N, M = 3001, 40
    w = synth.log_uniform_weights(N, seed=3, lo=1e-12)
    X = _field(N, M, 8, 1.0, np.float32 if prec else np.float64)
    p = pg.pod(_dev(X, torch.float32 if prec else torch.float64), w=torch.from_numpy(w).cuda(), remove_mean=False,
               energy=0.9, mode_kind=pg.MODES_PHYSICAL, prec=prec)
    eps = 2.0 ** -24 if prec else 2.0 ** -53
    _rows_agree(p.U.double().cpu().numpy(), np.sqrt(w)[:, None] * X, 2 * eps, 3, 1.0 / np.sqrt(w))


@pytest.mark.parametrize("small", [1e-8, 1e-12])
def test_rows_of_dmd_modes(small):
    N, M, K = 3000, 40, 6
    lam, amp = synth.oscillation_params(K, seed=3)
    D, _ = synth.oscillations(N, M, lam, amp, seed=4)
    scale = np.where(np.arange(N) % 3 == 1, small, 1.0)
    X = D * scale[:, None]
    a = pg.dmd(_dev(X), remove_mean=False, r_max=2 * K).Phi_packed.cpu().numpy()
    # every row of the modes is its row of the later snapshots times one matrix,
    # here from the large rows (reflectors do not keep small rows next to large
    # ones, so an explicit leaf height is no reference); perturbations of M eps
    # over the smallest kept value (1e-2 of the largest)
    rows = scale < 1.0
    C = np.linalg.lstsq(X[~rows, 1:], a[~rows], rcond=1e-9)[0]
    assert np.linalg.norm(a[rows] - X[rows, 1:] @ C) <= 1e-10 * np.linalg.norm(a[rows])


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("small_du", [False, True])
@pytest.mark.parametrize("N,M", [(2000, 30), (3000, 140)])
def test_rows_of_the_adjoint(N, M, small_du, prec):
    """dX of a Gram forward against its formula in numpy, which treats every row
    by itself, small rows alone and large ones (these against an explicit leaf
    height too); with cotangents that are small there too or not."""
    small = 1e-5 if prec else 1e-9
    dt = torch.float32 if prec else torch.float64
    s = 2.0 ** -np.arange(float(M))
    rng = np.random.default_rng(N)
    X = (rng.standard_normal((N, M)) * np.maximum(s, 1e-3)) @ synth.haar_orthogonal(M, 5).T
    rows = np.arange(N) % 3 == 1
    X[rows] *= small
    Xd = _dev(X, dt)
    g = torch.Generator(device="cuda")
    out, r = [], 4
    for b in (0, 1000):
        f = pg.pod(Xd, remove_mean=False, r_max=r, prec=prec, leaf_rows=b)
        dU = torch.randn((r, N), dtype=torch.float64, device="cuda", generator=g.manual_seed(1)).t() / N ** 0.5
        if small_du:
            dU[torch.from_numpy(rows).cuda()] *= small
        out.append(pg.pod_backward(f, (N, M), None, False, 0, b, r, dU=dU).cpu().numpy())
    Y, dU = Xd.double().cpu().numpy(), dU.cpu().numpy()
    _, S, gap = _modes(Y, r)
    VT = np.linalg.svd(Y, full_matrices=False)[2]
    VT *= np.sign(VT[np.arange(M), np.argmax(np.abs(VT), axis=1)])[:, None]
    A = VT @ (Y.T @ dU)                                      # v_i^T Y^T dU_j
    K = np.zeros((M, M))
    for i in range(M):
        for j in range(M):
            if i == j:
                K[i, i] = -A[i, i] / S[i] ** 3 if i < r else 0.0
            elif i < r or j < r:
                K[i, j] = ((A[i, j] / S[j] if j < r else 0.0) - (A[j, i] / S[i] if i < r else 0.0)) / (S[j] ** 2 - S[i] ** 2)
    ref = Y @ (VT.T @ K @ VT) + (dU / S[:r]) @ VT[:r]
    eps = 2.0 ** -24 if prec else 2.0 ** -53
    # kept values a factor of two apart, the last 1/8 of the first: 1e2 M eps
    for q in (rows, ~rows):
        assert np.linalg.norm(out[0][q] - ref[q]) <= 1e2 * M * eps * np.linalg.norm(ref[q])
    assert np.linalg.norm((out[0] - out[1])[~rows]) <= 1e2 * M * eps * np.linalg.norm(out[1][~rows])


@pytest.mark.parametrize("small", [0.05, 1e-3, 1e-5, 1e-8, 1e-30])
@pytest.mark.parametrize("shift", [0, 1])
def test_rows_of_batched_modes(small, shift):
    """Windows and bins of one plan, mixed precision; bins off a 16-byte boundary too."""
    wins = [_field(N, M, N, small, np.float32, zc) for N, M, zc in ((1500, 12, False), (801, 63, True), (2100, 96, False))]
    bins = []
    for N, M in ((1400, 20), (901, 70)):
        re, im = _field(N, M, N, small, np.float32), _field(N, M, N + 1, small, np.float32)
        im[2::3] *= small                                   # rows whose imaginary part is small
        bins.append(re + 1j * im.astype(np.float32))
    dev = []
    for Q in bins:
        big = torch.zeros((Q.shape[1], Q.shape[0] + shift), dtype=torch.complex64, device="cuda")
        big[:, shift:] = torch.from_numpy(np.ascontiguousarray(Q.T)).cuda()
        dev.append(big[:, shift:].t())
    b = pg.BatchedPOD([_dev(X, torch.float32) for X in wins], remove_mean=False, kmodes=3, prec=pg.PREC_MIXED_3XTF32,
                      bins=dev)
    b.run()
    assert b.status() == pg.OK
    eps = 2.0 ** -24
    for i, X in enumerate(wins):
        _rows_agree(b.modes[i].double().cpu().numpy(), X, eps, 3)
    for i, Q in enumerate(bins):
        U, S, VH = np.linalg.svd(Q, full_matrices=False)
        top = VH[np.arange(len(S)), np.argmax(np.abs(VH), axis=1)]
        V = (VH * (np.conj(top) / np.abs(top))[:, None]).conj().T
        gap = np.minimum(np.abs(np.diff(S, prepend=np.inf)), np.abs(np.diff(S, append=-np.inf)))
        got = b.modes[len(wins) + i].to(torch.complex128).cpu().numpy()
        rho = np.linalg.norm(Q, axis=1)
        for k in range(3):
            err = np.abs(got[:, k] - Q @ V[:, k] / S[k])[rho > 0] / (rho[rho > 0] / S[k])
            assert err.max() <= Q.shape[1] * eps * S[0] / gap[k], (i, k, err.max())


@pytest.mark.parametrize("spread", [2.0 ** -7, 2.0 ** -12, 2.0 ** -16])
def test_rows_of_batched_modes_with_uneven_columns(spread):
    """Columns within the spread that the shifts' short cut takes, and past it
    (further down the item is left to the Householder kernel)."""
    X = _field(1700, 24, 3, 1e-5, np.float32)
    X[:, ::2] *= spread
    X = X.astype(np.float32).astype(np.float64)
    b = pg.BatchedPOD([_dev(X, torch.float32)], remove_mean=False, kmodes=3, prec=pg.PREC_MIXED_3XTF32)
    b.run()
    assert b.status() == pg.OK
    _rows_agree(b.modes[0].double().cpu().numpy(), X, 2.0 ** -24, 3)
