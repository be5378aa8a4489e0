"""The work that users of this package have it do, as measurable cases.

Each case is one call (or one step) through the public entry points on inputs
that live on the GPU, from the shapes of quick looks at a small field to the
benchmark's 4,194,304 x 256 snapshot matrix:

  pod      the POD of a snapshot matrix (mean removal, cell volumes, binary64
           or 3xTF32 leaves, truncation by energy or to r_max modes)
  adjoint  one training step through the differentiable POD: forward,
           cotangents of modes and singular values, gradient of X
  dmd      exact DMD with optimal amplitudes
  spod     SPOD from the snapshots: block transforms, per-frequency SVDs, order
  bins     per-frequency complex SVDs of transforms that are already there
  windows  the PODs of several snapshot windows in one launch

Fields are what these methods meet: a smooth mean field, coherent structures
whose energy decays (43 of them hold 99 % of it, as in the benchmark's
spectrum) and a broadband floor.  The decompositions handed on are the
truncated ones: modes, right vectors of the kept modes, all singular values.
Paths whose leaves compute in binary32 hand their singular values and right
vectors on in binary32, the precision they have.
"""
import math

import numpy as np
import torch

import paper_2405_15529_gb300 as pg

DEV = "cuda"
FLOOR = 1e-5            # broadband floor under the coherent structures
ROW_CHUNK = 1 << 19


def listed():
    return [
        # a first look at a small field, as in an interactive session
        dict(name="pod_f64_4096x32", op="pod", N=4096, M=32, dtype="f64", prec="fp64", weights=False, mean=True,
             energy=0.99),
        # a plane cut with odd sizes, physical modes over uneven cells
        dict(name="pod_f64_65537x63", op="pod", N=65537, M=63, dtype="f64", prec="fp64", weights=True, mean=True,
             energy=0.99),
        # an ordinary volume field, all its modes kept up to 40
        dict(name="pod_f64_1048576x128", op="pod", N=1 << 20, M=128, dtype="f64", prec="fp64", weights=True,
             mean=True, energy=0.0, r_max=40),
        # the benchmark's workload
        dict(name="pod_f64_4194304x256", op="pod", N=1 << 22, M=256, dtype="f64", prec="fp64", weights=True,
             mean=False, energy=0.99),
        # binary32 snapshots of an ordinary and of a large field through the mixed path
        dict(name="pod_mixed_262144x100", op="pod", N=1 << 18, M=100, dtype="f32", prec="mixed", weights=False,
             mean=True, energy=0.99),
        dict(name="pod_mixed_4194304x256", op="pod", N=1 << 22, M=256, dtype="f32", prec="mixed", weights=True,
             mean=True, energy=0.99),
        # a long recording: many snapshots against the points
        dict(name="pod_mixed_300001x700", op="pod", N=300001, M=700, dtype="f32", prec="mixed", weights=False,
             mean=True, energy=0.99, r_max=128),
        # a training step of a reduced-order model
        dict(name="adjoint_f64_262144x64", op="adjoint", N=1 << 18, M=64, dtype="f64", prec="fp64", r=20, mean=True),
        # DMD of an oscillating wake
        dict(name="dmd_f64_524288x128", op="dmd", N=1 << 19, M=128, K=24, mean=True),
        # SPOD of a probe volume, windows of 64 with half overlap
        dict(name="spod_f32_131072x1056", op="spod", N=1 << 17, T=1056, npwin=64, nolap=32, kmodes=3),
        # frequency bins of uneven sizes, transforms made elsewhere
        dict(name="bins_24", op="bins", n=24, n_lo=1 << 14, n_hi=1 << 18, nb_lo=16, nb_hi=128, kmodes=4, prec="mixed"),
        # windows of a long run, each with its own mean and cells
        dict(name="windows_12", op="windows", n=12, n_lo=1 << 14, n_hi=1 << 18, nb_lo=16, nb_hi=96, kmodes=6,
             prec="mixed"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["pod", "pod", "pod", "mixed", "mixed", "adjoint", "dmd", "spod", "bins", "windows"])
    if op in ("pod", "mixed"):
        M = _log(rng, 16, 256 if op == "pod" else 700)
        N = _log(rng, max(4096, 4 * M), min(1 << 22, (1 << 37) // (M * M)))
        c = dict(op="pod", N=N, M=M, dtype="f32" if op == "mixed" else rng.choice(["f64", "f64", "f32"]),
                 prec="mixed" if op == "mixed" else "fp64", weights=rng.random() < 0.5, mean=rng.random() < 0.8)
        if rng.random() < 0.7:
            c["energy"] = rng.choice([0.9, 0.99])
        else:
            c.update(energy=0.0, r_max=max(2, min(M // 2, rng.randint(8, 48))))
        return c
    if op == "adjoint":
        M = _log(rng, 24, 128)
        mixed = rng.random() < 0.3
        return dict(op="adjoint", N=_log(rng, 8192, 1 << 19), M=M, dtype="f32" if mixed else "f64",
                    prec="mixed" if mixed else "fp64", r=rng.randint(4, min(20, M // 3)), mean=rng.random() < 0.5)
    if op == "dmd":
        K = rng.randint(6, 30)
        return dict(op="dmd", N=_log(rng, 16384, 1 << 20), M=rng.randint(2 * K + 8, 160), K=K,
                    mean=rng.random() < 0.5)
    if op == "spod":
        npwin = rng.choice([32, 48, 64, 64, 100])
        nolap = npwin // 2
        return dict(op="spod", N=_log(rng, 8192, 1 << 17), T=npwin + (npwin - nolap) * rng.randint(12, 40)
                    + rng.randint(0, 7), npwin=npwin, nolap=nolap, kmodes=3)
    n = rng.randint(4, 24 if op == "bins" else 12)
    lo = _log(rng, 1 << 13, 1 << 15)
    return dict(op=op, n=n, n_lo=lo, n_hi=lo * rng.randint(2, 8), nb_lo=16, nb_hi=rng.randint(24, 128 if op == "bins" else 96),
                kmodes=4 if op == "bins" else 6, prec="mixed" if rng.random() < 0.75 else "fp64")


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _randn(g, *shape, dtype=torch.float64):
    return torch.randn(shape, dtype=dtype, device=DEV, generator=g)


def _haar(g, M, dtype=torch.float64):
    """A Haar-distributed orthogonal (unitary) matrix, drawn on the device, its small QR on the host."""
    G = torch.randn((M, M), dtype=dtype, device=DEV, generator=g).cpu()
    Q, R = torch.linalg.qr(G)
    d = torch.diagonal(R)
    return (Q * (d / d.abs())[None, :]).to(DEV)


def _coherent(M):
    """Singular values of the field: six decades over 256, on the broadband floor."""
    i = torch.arange(M, dtype=torch.float64, device=DEV)
    return 10.0 ** (-6.0 * i / 255.0) + FLOOR


def _field(N, M, g, dtype, w, offset):
    """XT (M x N), its transpose the column-major snapshot matrix."""
    XT = torch.empty((M, N), dtype=dtype, device=DEV)
    mix = _coherent(M)[:, None] * _haar(g, M).T            # M x M
    for a in range(0, N, ROW_CHUNK):
        b = min(N, a + ROW_CHUNK)
        Y = mix.T @ _randn(g, M, b - a)                     # M x rows
        if w is not None:
            Y /= torch.sqrt(w[a:b])[None, :]
        if offset:
            x = torch.arange(a, b, dtype=torch.float64, device=DEV) * (2.0 * math.pi / N)
            Y += (1.0 + 0.5 * torch.cos(x))[None, :]
        XT[:, a:b] = Y
    return XT


def _cells(N, g):
    """Cell volumes, log-uniform over three decades."""
    return 10.0 ** (-3.0 * torch.rand(N, dtype=torch.float64, device=DEV, generator=g))


def _sizes(case):
    """Sizes of the bins or windows: spread log-uniformly in N and evenly in the columns, fixed by the case."""
    n = case["n"]
    out = []
    for i in range(n):
        u = ((i * 0.6180339887498949) % 1.0, (i + 0.5) / n)
        N = int(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** u[0])
        out.append((N, case["nb_lo"] + int(u[1] * (case["nb_hi"] - case["nb_lo"] + 1))))
    return out


def _dtype(name):
    return torch.float32 if name == "f32" else torch.float64


def _prec(name):
    return pg.PREC_MIXED_3XTF32 if name == "mixed" else pg.PREC_FP64


def _decay(M, g, cplx):
    """A decaying set of structures (each half the one before) on a small floor, mixed over the columns."""
    s = 2.0 ** -torch.arange(M, dtype=torch.float64, device=DEV) + 1e-3
    dt = torch.complex128 if cplx else torch.float64
    return s.to(dt)[:, None] * _haar(g, M, dt)


def _inputs(case, seed):
    g = _gen(seed)
    op = case["op"]
    if op in ("pod", "adjoint"):
        w = _cells(case["N"], g) if case.get("weights") else None
        XT = _field(case["N"], case["M"], g, _dtype(case["dtype"]), w, case["mean"])
        d = dict(X=XT.t(), w=w)
        if op == "adjoint":
            d["gU"] = _randn(g, case["r"], case["N"]).t().to(_dtype(case["dtype"])) / math.sqrt(case["N"])
            d["gS"] = _randn(g, case["M"])
            d["gS"][case["r"]:] = 0.0
        return d
    if op == "dmd":
        N, M, K = case["N"], case["M"], case["K"]
        k = torch.arange(K, dtype=torch.float64, device=DEV)
        rho = 0.985 + 0.015 * torch.rand(K, dtype=torch.float64, device=DEV, generator=g)
        ph = 2.0 * math.pi * torch.rand(K, dtype=torch.float64, device=DEV, generator=g)
        t = torch.arange(M, dtype=torch.float64, device=DEV)
        C = ((1.0 + k / K) * torch.exp(1j * ph))[:, None] * torch.polar(
            rho[:, None] ** t[None, :], (0.05 + 2.95 * k / max(K - 1, 1))[:, None] * t[None, :])
        XT = torch.empty((M, N), dtype=torch.float64, device=DEV)
        for a in range(0, N, ROW_CHUNK):
            b = min(N, a + ROW_CHUNK)
            XT[:, a:b] = C.real.T @ _randn(g, K, b - a) - C.imag.T @ _randn(g, K, b - a) + 0.5
            XT[:, a:b] += 1e-5 * _randn(g, M, b - a)
        return dict(X=XT.t())
    if op == "spod":
        N, T = case["N"], case["T"]
        J = 8
        a = 2.0 ** -torch.arange(J, dtype=torch.float32, device=DEV)
        D = (a[:, None] * _randn(g, J, T, dtype=torch.float32)).T @ _randn(g, J, N, dtype=torch.float32)   # T x N
        D += 1e-3 * _randn(g, T, N, dtype=torch.float32)
        D += 1.0
        return dict(X=D.t())
    if op == "bins":
        Q = []
        for N, Nb in _sizes(case):
            G = torch.randn((Nb, N), dtype=torch.complex64, device=DEV, generator=g)
            Q.append((_decay(Nb, g, True).to(torch.complex64).T @ G / math.sqrt(Nb)).t())
        return dict(Q=Q)
    X, w = [], []
    for i, (N, M) in enumerate(_sizes(case)):
        wi = _cells(N, g) if i % 2 == 0 else None
        Y = _decay(M, g, False).T @ _randn(g, M, N)
        if wi is not None:
            Y /= torch.sqrt(wi)[None, :]
        dt = torch.float32 if case["prec"] == "mixed" else torch.float64
        X.append((Y + 1.0).to(dt).t())
        w.append(wi)
    return dict(X=X, w=w)


# ---------------------------------------------------------------- the calls

def prepare(case, seed):
    """Inputs on the GPU and what a program keeps between calls: the workspace
    of the repeated POD and DMD, the plan of the batched launches."""
    s = dict(_inputs(case, seed), case=case)
    op = case["op"]
    if op == "pod":
        N, M = s["X"].shape
        need = pg.pod_workspace_size(N, M, r_max=case.get("r_max"),
                                     xtype=pg.F32 if case["dtype"] == "f32" else pg.F64, prec=_prec(case["prec"]))
        s["ws"] = torch.empty(need, dtype=torch.uint8, device=DEV)
    elif op == "adjoint":
        s["X"].requires_grad_(True)
    elif op == "dmd":
        N, M = s["X"].shape
        s["ws"] = torch.empty(pg.dmd_workspace_size(N, M, r_max=2 * case["K"]), dtype=torch.uint8, device=DEV)
    elif op == "spod":
        s["plan"] = pg.SPOD(s["X"], dt=0.2, npwin=case["npwin"], nolap=case["nolap"], kmodes=case["kmodes"])
    elif op == "bins":
        s["plan"] = pg.BatchedSVD(s["Q"], kmodes=case["kmodes"], prec=_prec(case["prec"]))
    else:
        s["plan"] = pg.BatchedPOD(s["X"], weights=s["w"], kmodes=case["kmodes"], prec=_prec(case["prec"]))
    return s


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "pod":
        p = pg.pod(s["X"], w=s["w"], remove_mean=case["mean"], energy=case["energy"], r_max=case.get("r_max"),
                   prec=_prec(case["prec"]), workspace=s["ws"])
        V = p.VT[:p.r]
        if case["prec"] == "mixed":
            return dict(U=p.U, S=p.S.float(), VT=V.float(), mean=p.mean)
        return dict(U=p.U, S=p.S, VT=V, mean=p.mean)
    if op == "adjoint":
        U, S, VT = pg.pod_autograd(s["X"], case["r"], remove_mean=case["mean"], prec=_prec(case["prec"]))
        dX, = torch.autograd.grad((U, S), (s["X"],), (s["gU"], s["gS"]))
        if case["prec"] == "mixed":
            return dict(U=U, S=S.float(), VT=VT[:case["r"]].float(), dX=dX)
        return dict(U=U, S=S, VT=VT[:case["r"]], dX=dX)
    if op == "dmd":
        d = pg.dmd(s["X"], remove_mean=case["mean"], r_max=2 * case["K"], workspace=s["ws"])
        return dict(mu=d.mu, b=d.b, Phi=d.Phi_packed, S=d.S)
    p = s["plan"]
    p.run()
    if op == "spod":
        return dict(L=p.L.float(), order=p.order, modes=p.modes)
    S = p.S_all.float() if case["prec"] == "mixed" else p.S_all
    if op == "bins":
        return dict(S=S, modes=p.modes)
    return dict(S=S, modes=p.modes, VT=[v[:k].float() if case["prec"] == "mixed" else v[:k] for v, k in zip(p.VT, p.k)],
                mean=p.mean)


# ---------------------------------------------------------------- bytes and operations

def _kept(M, energy, r_max):
    """Modes that an energy share keeps of the field's spectrum."""
    if energy <= 0.0:
        return r_max or M
    e = np.cumsum((10.0 ** (-6.0 * np.arange(M) / 255.0) + FLOOR) ** 2)
    return min(int(np.searchsorted(e, energy * e[-1])) + 1, r_max or M)


def work(case):
    """Inputs read once, outputs written once; operations of an R factor (2 N M^2), the modes of the kept
    directions (2 N M r) and, for the adjoint, the two products of the gradient."""
    op = case["op"]
    if op in ("pod", "adjoint"):
        N, M = case["N"], case["M"]
        b = 4 if case["dtype"] == "f32" else 8
        bo = 4 if case["prec"] == "mixed" else 8
        if op == "pod":
            r = _kept(M, case["energy"], case.get("r_max"))
            return dict(bytes=N * (M * b + r * bo + 8 + (8 if case["weights"] else 0)), flops=2.0 * N * M * M + 2.0 * N * M * r)
        r = case["r"]
        return dict(bytes=N * (2 * M * b + 2 * r * bo), flops=2.0 * N * M * M + 2.0 * N * M * r + 4.0 * N * M * r + 2.0 * N * M * M)
    if op == "dmd":
        N, M, r = case["N"], case["M"], 2 * case["K"]
        return dict(bytes=8 * N * (M + r + 1), flops=2.0 * N * M * M + 2.0 * N * M * r)
    if op == "spod":
        N, T = case["N"], case["T"]
        nb = (T - case["nolap"]) // (case["npwin"] - case["nolap"])
        nf = case["npwin"] // 2 + 1
        fft = 2.5 * case["npwin"] * math.log2(case["npwin"]) * nb * N
        return dict(bytes=4 * N * T + 8 * N * nf * case["kmodes"], flops=fft + nf * 8.0 * N * nb * (nb + case["kmodes"]))
    k, real = case["kmodes"], op == "windows"
    b = 8 if (not real or case["prec"] != "mixed") else 4
    c = 2.0 if real else 8.0
    return dict(bytes=sum(b * N * (M + k) for N, M in _sizes(case)), flops=sum(c * N * M * (M + k) for N, M in _sizes(case)))


# ---------------------------------------------------------------- the same in 64 bits, by library routines

def _svd_tall(Y, k):
    """Singular values, first k left and right vectors of a tall matrix, the largest entry of each right
    vector made real and positive: a QR of row blocks, an SVD of the small factor."""
    M = Y.shape[1]
    R = None
    for a in range(0, Y.shape[0], 1 << 18):
        blk = Y[a:a + (1 << 18)]
        R = torch.linalg.qr(blk if R is None else torch.cat([R, blk]), mode="r")[1]
    _, S, Vh = np.linalg.svd(R.cpu().numpy())
    S = np.concatenate([S, np.zeros(M - S.shape[0])])
    V = Vh.conj().T
    j = np.argmax(np.abs(V), axis=0)
    e = V[j, np.arange(M)]
    V = V * (e.conj() / np.abs(e))[None, :]
    S, V = torch.tensor(S, device=DEV), torch.tensor(np.ascontiguousarray(V), device=DEV)
    return (Y @ V[:, :k]) / S[:k].to(Y.dtype), S, V


def _exact_pod(X, w, mean, k):
    X = X.detach().double()
    m = X.mean(dim=1) if mean else torch.zeros(X.shape[0], dtype=torch.float64, device=DEV)
    Y = X - m[:, None]
    if w is not None:
        Y *= torch.sqrt(w)[:, None]
    return (m, Y) + _svd_tall(Y, k)


def _exact_adjoint(case, d):
    X, r = d["X"], case["r"]
    M = X.shape[1]
    m, Y, U, S, V = _exact_pod(X, None, case["mean"], M)
    k = M - 1 if case["mean"] else M                    # directions that the removed mean leaves
    U, Sk, Vk = U[:, :k], S[:k], V[:, :k]
    gU = torch.zeros((X.shape[0], k), dtype=torch.float64, device=DEV)
    gU[:, :r] = d["gU"].double()
    D = (Sk[None, :] - Sk[:, None]) * (Sk[None, :] + Sk[:, None])
    D.fill_diagonal_(1.0)
    F = 1.0 / D
    F.fill_diagonal_(0.0)
    Z = U.T @ gU
    K = (F * (Z - Z.T)) * Sk[None, :] + torch.diag(d["gS"][:k])
    dY = U @ (K @ Vk.T) + ((gU - U @ Z) / Sk[None, :]) @ Vk.T
    if case["mean"]:
        dY -= dY.mean(dim=1, keepdim=True)
    return dict(U=U[:, :r], S=S, VT=V[:, :r].T, dX=dY)


def _exact_dmd(case, d):
    X = d["X"]
    N, M = X.shape
    r = 2 * case["K"]
    m = X.mean(dim=1) if case["mean"] else torch.zeros(N, dtype=torch.float64, device=DEV)
    Y = X - m[:, None]
    U, S, V = _svd_tall(Y[:, :-1], r)
    Sr, Vr = S[:r].cpu().numpy(), V[:, :r].cpu().numpy()
    A = (U.T @ Y[:, 1:]).cpu().numpy() @ (Vr / Sr[None, :])
    mu, W = np.linalg.eig(A)
    W = W / np.linalg.norm(W, axis=0)[None, :]
    p = W[np.argmax(np.abs(W), axis=0), np.arange(r)]
    W = W * (p.conj() / np.abs(p))[None, :]
    Vand = mu[:, None] ** np.arange(M - 1)[None, :]
    P = (W.conj().T @ W) * np.conj(Vand @ Vand.conj().T)
    q = np.conj(np.diag(Vand @ (Vr * Sr[None, :]) @ W))
    b = np.linalg.solve(P, q)
    key = np.array([max(abs(b[i]), abs(b[np.argmin(np.abs(mu - mu[i].conj()))])) for i in range(r)])
    pair = np.array([min(i, int(np.argmin(np.abs(mu - mu[i].conj())))) for i in range(r)])
    idx = sorted(range(r), key=lambda i: (-key[pair[i]], pair[i], -mu[i].imag))
    mu, b, W = mu[idx], b[idx], W[:, idx]
    Phi = Y[:, 1:].to(torch.complex128) @ torch.tensor((Vr / Sr[None, :]) @ W / mu[None, :], device=DEV)
    packed = torch.where(torch.tensor(mu.imag < 0, device=DEV)[None, :], torch.roll(Phi.imag, 1, dims=1), Phi.real)
    return dict(mu=torch.tensor(mu), b=torch.tensor(b), Phi=packed, S=S)


def _exact_spod(case, d):
    D = d["X"].double()
    n, hop = case["npwin"], case["npwin"] - case["nolap"]
    nb, nf = (D.shape[1] - case["nolap"]) // hop, n // 2 + 1
    D = D - D.mean(dim=1, keepdim=True)
    j = torch.arange(n, dtype=torch.float64, device=DEV)
    win = 0.54 - 0.46 * torch.cos(2.0 * math.pi * j / (n - 1))
    scale = torch.full((nf,), 2.0, dtype=torch.float64, device=DEV)
    scale[0] = scale[-1] = 1.0
    scale /= win.sum() * math.sqrt(nb)
    Q = torch.empty((nf, nb, D.shape[0]), dtype=torch.complex128, device=DEV)
    for b in range(nb):
        Q[:, b] = (torch.fft.rfft(D[:, b * hop:b * hop + n] * win[None, :], dim=1) * scale[None, :]).T
    L, U = [], []
    for f in range(nf):
        u, s, _ = _svd_tall(Q[f].t(), case["kmodes"])
        L.append(s ** 2)
        U.append(u)
    L = torch.stack(L)
    return dict(L=L, order=torch.argsort(L[:, 0], descending=True, stable=True), modes=U)


def exact(case, seed):
    d = _inputs(case, seed)
    op = case["op"]
    if op == "pod":
        M = case["M"]
        k = _kept(M, case["energy"], case.get("r_max"))
        m, Y, U, S, V = _exact_pod(d["X"], d["w"], case["mean"], M if case["energy"] > 0 else k)
        if case["energy"] > 0:
            e = torch.cumsum(S ** 2, 0)
            k = min(int((e < case["energy"] * e[-1]).sum()) + 1, case.get("r_max") or M)
        return dict(U=U[:, :k], S=S, VT=V[:, :k].T, mean=m)
    if op == "adjoint":
        return _exact_adjoint(case, d)
    if op == "dmd":
        return _exact_dmd(case, d)
    if op == "spod":
        return _exact_spod(case, d)
    out = dict(S=[], modes=[])
    if op == "bins":
        for Q in d["Q"]:
            U, S, _ = _svd_tall(Q.to(torch.complex128), min(case["kmodes"], Q.shape[1]))
            out["S"].append(S)
            out["modes"].append(U)
    else:
        out.update(VT=[], mean=[])
        for X, w in zip(d["X"], d["w"]):
            k = min(case["kmodes"], X.shape[1])
            m, _, U, S, V = _exact_pod(X, w, True, k)
            out["S"].append(S)
            out["modes"].append(U)
            out["VT"].append(V[:, :k].T)
            out["mean"].append(m)
    out["S"] = torch.cat(out["S"])
    return out
