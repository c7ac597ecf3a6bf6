"""Workloads that a user of the eigensolver runs, through its public entry points.

Families:
  apply    Solver.apply_H on a block of bands (kinetic + FFT local potential + KB projectors)
  gemm_nn  tall products A B: Ritz updates, rotations, constraint and KB back-projections
  gemm_cn  long reductions A^H B: Gram blocks, constraint and KB projections
  gram     lower triangle of a Hermitian Gram matrix in the FP64 class
  rr       one Rayleigh-Ritz step and the density matrix of its occupied bands
  solve    lowest eigenpairs from random start vectors, then the electron density

The cells are synthetic: Gaussian atoms on jittered sites, s + p Gaussian KB projectors, random
normal bands that fall off with the kinetic energy.  Everything is made from the seed on the GPU.
"""
import math

import numpy as np
import torch

import paper_0707_3405_gb300 as lg

DEV = "cuda"
C128, C64, F64 = torch.complex128, torch.complex64, torch.float64


# ------------------------------------------------------------------ which cases
def listed():
    return [
        # one small Gamma cell: the H application of a molecule-sized job, a few launches long
        dict(name="apply_c64_n24", family="apply", prec="c64", a=10.0, N=24, nat=4, nproj=0, kx=0.0, nb=16),
        # H W of one inner iteration of the mixed schedule on a 108-atom cell
        dict(name="apply_c64_n120", family="apply", prec="c64", a=25.0, N=120, nat=108, nproj=432, kx=0.0, nb=128),
        # the FP64-class H X refresh of one block of the same cell
        dict(name="apply_tc_n120", family="apply", prec="tc", a=25.0, N=120, nat=108, nproj=432, kx=0.0, nb=128),
        # H X of one block in plain FP64 (the default schedule) at a general k-point
        dict(name="apply_c128_n72", family="apply", prec="c128", a=16.0, N=72, nat=32, nproj=128, kx=0.125, nb=64),
        # P = [W P] C of the mixed schedule
        dict(name="nn_c64_update", family="gemm_nn", prec="c64", M=113081, n=128, k=256, beta=0.0),
        # all-band Ritz rotation closing a sweep of a 256 + 64 band solve, FP64 class
        dict(name="nn_tc_rotation", family="gemm_nn", prec="tc", M=57925, n=320, k=320, beta=0.0),
        # Y^H X_b, the constraint of a block start against four earlier blocks, FP64 class.  (The
        # complex64 reductions are in apply and solve: their FP32 sums over 1e5 terms round by up
        # to 1e-4 of the result, which the later steps forgive.)
        dict(name="cn_tc_constraint", family="gemm_cn", prec="tc", m=512, n=128, K=113081),
        # Gram matrix closing a sweep of a 1024 + 128 band solve, FP64 class
        dict(name="gram_tc_1152", family="gram", prec="tc", n=1152, K=113081),
        # Rayleigh-Ritz on [X W P] of a 128-band block: one of these per inner iteration
        dict(name="rr_df32_384", family="rr", prec="df32", n=384, m=128),
        # all-band Rayleigh-Ritz closing a sweep of a 1024 + 128 band solve
        dict(name="rr_df32_1152", family="rr", prec="df32", n=1152, m=1152),
        # whole solve of a small cell in FP64
        dict(name="solve_fp64_n24", family="solve", prec="fp64", a=10.0, N=24, nat=4, nproj=0, kx=0.0, M=16, block=16),
        # whole mixed-precision solve of a 64-atom cell
        dict(name="solve_mixed_n96", family="solve", prec="mixed", a=20.0, N=96, nat=64, nproj=256, kx=0.25, M=256,
             block=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["apply", "apply", "gemm_nn", "gemm_cn", "gram", "rr", "solve"])
    if family == "apply":
        prec = rng.choice(["c64", "c64", "tc", "df32", "c128"])
        N = rng.choice([18, 20, 24, 30, 36, 40, 45, 48, 54, 60, 64, 72, 80, 90, 96, 100, 108, 120, 128])
        nat = rng.randint(0, max(1, (N // 8) ** 3 // 24))
        work = (N / 120.0) ** 3 * {"c64": 1.0, "tc": 1.0, "df32": 1.0, "c128": 4.0}[prec]
        nb = _log(rng, 1, max(2, min(256, 128 / work)))
        return dict(family=family, prec=prec, a=round(N * rng.uniform(0.2, 0.24), 3), N=N, nat=max(nat, 1),
                    nproj=4 * nat, kx=rng.choice([0.0, 0.125, 0.25, 0.375]), nb=nb)
    if family == "gemm_nn":
        prec = rng.choice(["c64", "c64", "tc", "tc", "df32", "c128"])
        top = 384 if prec in ("c64", "tc") else 96
        return dict(family=family, prec=prec, M=_log(rng, 900, 120000), n=_log(rng, 8, top),
                    k=_log(rng, 8, top + top // 3), beta=rng.choice([0.0, 1.0]))
    if family == "gemm_cn":
        prec = rng.choice(["c64", "tc", "tc", "df32", "c128"])
        top = 512 if prec in ("c64", "tc") else 96
        return dict(family=family, prec=prec, m=_log(rng, 8, top), n=_log(rng, 8, top),
                    K=_log(rng, 900, 6000 if prec == "c64" else 120000))
    if family == "gram":
        return dict(family=family, prec="tc", n=_log(rng, 16, 1000), K=_log(rng, 900, 110000))
    if family == "rr":
        n = _log(rng, 24, 900)
        m = n if rng.random() < 0.4 else max(1, n // 3)
        return dict(family=family, prec=rng.choice(["df32", "df32", "fp64"]), n=n, m=m)
    N = rng.choice([20, 24, 30, 32, 36])
    block = rng.choice([8, 12, 16, 20])
    nat = rng.randint(3, 6)
    return dict(family="solve", prec=rng.choice(["mixed", "fp64"]), a=round(N * rng.uniform(0.3, 0.42), 3), N=N, nat=nat,
                nproj=4 * nat * rng.randint(0, 1), kx=rng.choice([0.0, 0.125, 0.25]), M=block * rng.randint(1, 3),
                block=block)


# ------------------------------------------------------------------ synthetic cells
def _rng(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape):
    return torch.randn(*shape, dtype=F64, device=DEV, generator=g)


def _rand(g, *shape):
    return torch.rand(*shape, dtype=F64, device=DEV, generator=g)


def _crandn(g, *shape):
    return torch.complex(_randn(g, *shape), _randn(g, *shape)) * math.sqrt(0.5)


def _ecut(case):
    return 0.5 * (math.pi * case["N"] / (2.0 * case["a"])) ** 2


def _sphere(case):
    """Miller indices (npw, 3) of the plane waves in the library's documented order."""
    a, N, kx = case["a"], case["N"], case["kx"]
    r2 = 2.0 * _ecut(case) * (a / (2.0 * math.pi)) ** 2
    lim = int(math.ceil(math.sqrt(r2))) + 2
    n = torch.arange(-lim, lim + 1, dtype=F64, device=DEV) + kx
    inside = (n[:, None, None] ** 2 + n[None, :, None] ** 2) + n[None, None, :] ** 2 <= r2 + 1e-9
    return torch.nonzero(inside) - lim


def _cell(case, g):
    """Atoms, V(r) on the grid and, where the case has projectors, their energies."""
    a, N, nat = case["a"], case["N"], case["nat"]
    side = max(1, math.ceil(nat ** (1.0 / 3.0) - 1e-9))
    sites = torch.cartesian_prod(*[torch.arange(side, dtype=F64, device=DEV)] * 3).reshape(-1, 3)
    pick = torch.randperm(len(sites), device=DEV, generator=g)[:nat]
    pos = (sites[pick] + 0.5 + (0.3 * _rand(g, nat, 3) - 0.15)) * (a / side)
    depth = -3.0 + 2.0 * _rand(g, nat)
    width = 0.8 + 0.4 * _rand(g, nat)
    i = torch.arange(N, device=DEV)
    gx = (2.0 * math.pi / a) * torch.where(i < (N + 1) // 2, i, i - N).to(F64)
    f = [torch.exp(torch.complex(-0.5 * width[:, None] ** 2 * gx[None, :] ** 2, -gx[None, :] * pos[:, d, None]))
         for d in range(3)]
    if N % 2 == 0:  # no Nyquist planes
        for x in f:
            x[:, N // 2] = 0.0
    pref = depth * (2.0 * math.pi * width ** 2) ** 1.5 / a ** 3
    xy = (pref[:, None, None] * f[0][:, :, None] * f[1][:, None, :]).reshape(nat, N * N)
    vhat = (xy.T @ f[2]).reshape(N, N, N)
    v = (torch.fft.ifftn(vhat).real * float(N ** 3)).contiguous()
    E = None
    if case["nproj"]:
        e = -1.0 + 2.0 * _rand(g, nat, 2)
        E = torch.stack([e[:, 0], e[:, 1], e[:, 1], e[:, 1]], dim=1).reshape(-1)
    return pos, v, E


def _beta(case, mil, pos):
    """KB projectors, (nproj, npw): one row per projector."""
    a = case["a"]
    q = (2.0 * math.pi / a) * (mil.to(F64) + case["kx"])
    c = (4.0 * math.pi) ** 0.75 / math.sqrt(a ** 3)
    radial = c * torch.exp(-0.5 * (q * q).sum(1))
    ph = torch.exp(torch.complex(torch.zeros_like(pos @ q.T), -(pos @ q.T))) * radial
    p = [math.sqrt(2.0) * q[:, d] * ph for d in range(3)]
    return torch.stack([ph] + p, dim=1).reshape(case["nproj"], len(mil))


def _kin(case, mil):
    q = (2.0 * math.pi / case["a"]) * (mil.to(F64) + case["kx"])
    return 0.5 * (q * q).sum(1)


def _bands(case, mil, nb, g):
    x = _crandn(g, nb, len(mil)) / (1.0 + _kin(case, mil))
    return x / torch.linalg.vector_norm(x, dim=1, keepdim=True)


def _solver(case, pos, v, E, **kw):
    beta = None
    if E is not None:
        def beta(mil, k):
            return _beta(case, torch.from_numpy(mil.astype(np.int64)).to(DEV), pos).cpu().numpy().T
    return lg.Solver(case["a"], case["N"], _ecut(case), [[case["kx"]] * 3], v.cpu().numpy(),
                     None if E is None else E.cpu().numpy(), beta=beta, **kw)


# ------------------------------------------------------------------ matrices
def _columns(g, cols, rows, prec):
    """A block of bands as stored: (cols, rows), columns of norm about one that fall off with the
    row like plane-wave coefficients do over the sphere."""
    d = 1.0 / (1.0 + 4.0 * torch.rand(rows, dtype=F64, device=DEV, generator=g) ** 2)
    x = _crandn(g, cols, rows) * (d * (1.6 / math.sqrt(rows)))
    return x.to(C64) if prec == "c64" else x


def _overlapping(g, a, n, prec):
    """n columns that overlap with those of ``a`` as the factors of a Gram block or of a projection
    do: [W P] are columns of [R W P] themselves, W is K R, a projector sits where the bands are."""
    i = torch.arange(len(a) - n, len(a), device=DEV) % len(a)
    return (0.8 * a[i] + 0.6 * _columns(g, n, a.shape[1], prec)).to(a.dtype)


def _pencil(g, n, m):
    """S and A of a Rayleigh-Ritz step, and the occupation function (mu, T) of its bands."""
    def herm(k):
        h = _crandn(g, k, k)
        return (h + h.mH) * (0.5 / math.sqrt(k))

    theta = torch.sort(-1.0 + 1.5 * _rand(g, m))[0]
    if m == n:  # all bands of a sweep: nearly orthonormal, nearly diagonal
        S = torch.eye(n, dtype=C128, device=DEV) + 1e-6 * herm(n)
        A = torch.diag(theta).to(C128) + 1e-3 * herm(n)
    else:       # [X W P]: X orthonormal and diagonal, W and P correlated and weakly coupled to X
        r = n - m
        S = torch.eye(n, dtype=C128, device=DEV)
        T = torch.eye(r, dtype=C128, device=DEV) + 0.4 * _crandn(g, r, r) / math.sqrt(r)
        T = T / torch.linalg.vector_norm(T, dim=0, keepdim=True)
        S[m:, m:] = T.mH @ T
        A = torch.zeros(n, n, dtype=C128, device=DEV)
        A[:m, :m] = torch.diag(theta).to(C128)
        h = torch.sort(1.0 + 5.0 * _rand(g, r))[0]
        A[m:, m:] = T.mH @ (h.to(C128)[:, None] * T)
        A[m:, :m] = 0.02 * _crandn(g, r, m)
        A[:m, m:] = A[m:, :m].mH
    S = 0.5 * (S + S.mH)
    A = 0.5 * (A + A.mH)
    return S, A, -0.25, 0.0375


def _prec_kw(prec):
    return dict(df32=prec == "df32", tc=prec == "tc")


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    g = _rng(seed)
    fam = case["family"]
    st = {"case": case}
    if fam in ("apply", "solve"):
        pos, v, E = _cell(case, g)
        mil = _sphere(case)
        if fam == "apply":
            st["solver"] = _solver(case, pos, v, E, block_size=max(1, case["nb"]))
            x = _bands(case, mil, case["nb"], g)
            st["X"] = x.to(C64) if case["prec"] == "c64" else x
            st["Y"] = torch.empty_like(st["X"])
        else:
            st["solver"] = _solver(case, pos, v, E, block_size=case["block"], nline=4, max_sweeps=100,
                                   precision=case["prec"], tol=1e-8, nbuf=case["block"], use_graph=True)
            st["X0"] = _crandn(g, case["M"], len(mil))
    elif fam == "gemm_nn":
        st["A"] = _columns(g, case["k"], case["M"], case["prec"])
        b = _crandn(g, case["n"], case["k"]) / math.sqrt(case["k"])
        st["B"] = b.to(C64) if case["prec"] == "c64" else b
        st["C"] = _columns(g, case["n"], case["M"], case["prec"]) if case["beta"] else None
        st["D"] = torch.empty(case["n"], case["M"], dtype=st["A"].dtype, device=DEV)
    elif fam == "gemm_cn":
        st["A"] = _columns(g, case["m"], case["K"], case["prec"])
        st["B"] = _overlapping(g, st["A"], case["n"], case["prec"])
        st["C"] = torch.empty(case["n"], case["m"], dtype=st["A"].dtype, device=DEV)
    elif fam == "gram":
        st["A"] = _columns(g, case["n"], case["K"], case["prec"])
        st["C"] = torch.zeros(case["n"], case["n"], dtype=C128, device=DEV)
    else:
        S, A, st["mu"], st["T"] = _pencil(g, case["n"], case["m"])
        st["S"], st["A"] = S.T.contiguous(), A.T.contiguous()  # stored column-major
    return st


def run(st):
    case = st["case"]
    fam, prec = case["family"], case["prec"]
    if fam == "apply":
        return st["solver"].apply_H(0, st["X"], st["Y"], **_prec_kw(prec))
    if fam == "gemm_nn":
        return lg.gemm_nn(st["A"], st["B"], 1.0, case["beta"], st["C"], st["D"], **_prec_kw(prec))
    if fam == "gemm_cn":
        return lg.gemm_cn(st["A"], st["B"], C=st["C"], **_prec_kw(prec))
    if fam == "gram":
        return lg.gram_lower(st["A"], st["A"], C=st["C"], **_prec_kw(prec))
    if fam == "rr":
        # A Ritz vector is free up to its phase, and close ones mix: the density matrix of the
        # occupied bands is the quantity that is not, and what a density or an energy is made of
        theta, C, _ = lg.rayleigh_ritz(st["S"], st["A"], case["m"], df32=prec == "df32")
        f = torch.sigmoid((st["mu"] - theta) / st["T"])
        occ = (f[:, None] * C.conj()).T.contiguous()
        return {"theta": theta, "rho": lg.gemm_nn(C, occ, tc=True)}
    X = st["X0"].clone()
    res = st["solver"].solve(X)
    # occupations that vanish at the highest bands, and the density in FP32 as it is stored: the
    # bands are converged to about 1e-6, and their phases are free
    f, e = _occupations(res.eig[0])
    rho = st["solver"].density(0, X, f, df32=True)
    return {"eig": e, "rho": rho.to(torch.float32)}


def _occupations(e):
    mid = len(e) // 2
    mu = 0.5 * (e[mid - 1] + e[mid])
    T = max((e[-1] - mu) / 20.0, 1e-3)
    return 2.0 / (1.0 + np.exp(np.minimum((e - mu) / T, 700.0))), np.array(e)


# ------------------------------------------------------------------ what a pass cannot do without
def _npw(case):
    return 4.0 / 3.0 * math.pi * (case["N"] / 4.0) ** 3


def _apply_work(case, nb):
    N, npw, el = case["N"], _npw(case), 8 if case["prec"] in ("c64", "mixed") else 16
    # sphere -> grid -> sphere with the empty rows and planes left out: z-lines inside the sphere's
    # disc, y-lines on its x-planes, all x-lines, each forward and back
    lines = math.pi * (N / 4.0) ** 2 + N * N / 2.0 + N * N
    fl = nb * (2.0 * lines * 5.0 * N * math.log2(N) + 8.0 * N ** 3 / 4.0 + 16.0 * npw * case["nproj"])
    by = el * npw * (2.0 * nb + case["nproj"]) + el / 2.0 * (N ** 3 + npw)
    return by, fl


def work(case):
    fam = case["family"]
    el = 8 if case["prec"] == "c64" else 16
    if fam == "apply":
        by, fl = _apply_work(case, case["nb"])
    elif fam == "gemm_nn":
        M, n, k = case["M"], case["n"], case["k"]
        by, fl = el * (M * k + k * n + M * n * (2.0 if case["beta"] else 1.0)), 8.0 * M * n * k
    elif fam == "gemm_cn":
        m, n, K = case["m"], case["n"], case["K"]
        by, fl = el * (K * (m + n) + m * n), 8.0 * K * m * n
    elif fam == "gram":
        n, K = case["n"], case["K"]
        by, fl = el * (K * n + n * n / 2.0), 4.0 * K * n * n
    elif fam == "rr":
        n, m = case["n"], case["m"]
        by = 16.0 * (2.0 * n * n + n * n)
        fl = 8.0 * (n ** 3 / 3.0 + n ** 3 + 4.0 / 6.0 * n ** 3 + n * n * m + n * n * m + n * n * m)
    else:  # one sweep of nline = 4 iterations over every block and its closing step, five times
        M, m = case["M"] + case["block"], case["block"]
        by, fl = _apply_work(case, M)
        npw = _npw(case)
        inner = 8.0 * npw * M * (2.0 * M + 4.0 * m + 3.0 * m + 2.0 * m + 8.0 * m)
        by = 5 * (5 * by + 16.0 * npw * M * 4)
        fl = 5 * (5 * fl + 4 * inner + 24.0 * npw * M * M)
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ the same in 64 bits
def _h_apply(case, mil, v, E, beta, x):
    """H x for bands x (nb, npw) by library transforms in FP64."""
    N = case["N"]
    idx = mil % N
    flat = (idx[:, 0] * N + idx[:, 1]) * N + idx[:, 2]
    y = x * _kin(case, mil)
    step = max(1, int(2e9 // (16 * N ** 3)))
    for b in range(0, len(x), step):
        box = torch.zeros(len(x[b:b + step]), N ** 3, dtype=C128, device=DEV)
        box[:, flat] = x[b:b + step]
        box = box.reshape(-1, N, N, N)
        box = torch.fft.fftn(torch.fft.ifftn(box, dim=(1, 2, 3)) * v, dim=(1, 2, 3))
        y[b:b + step] += box.reshape(-1, N ** 3)[:, flat]
    if E is not None:
        y += ((x @ beta.mH) * E) @ beta
    return y


def exact(case, seed):
    g = _rng(seed)
    fam, prec = case["family"], case["prec"]
    if fam in ("apply", "solve"):
        pos, v, E = _cell(case, g)
        mil = _sphere(case)
        beta = None if E is None else _beta(case, mil, pos)
        if fam == "apply":
            x = _bands(case, mil, case["nb"], g)
            x = x.to(C64).to(C128) if prec == "c64" else x
            return _h_apply(case, mil, v, E, beta, x)
        if len(mil) > 2000:
            return None
        h = _h_apply(case, mil, v, E, beta, torch.eye(len(mil), dtype=C128, device=DEV)).cpu().numpy().T
        e, u = np.linalg.eigh(0.5 * (h + h.conj().T))
        M, N = case["M"], case["N"]
        f, e = _occupations(e[:M])
        u = torch.from_numpy(np.ascontiguousarray(u[:, :M].T)).to(DEV)
        idx = mil % N
        box = torch.zeros(M, N ** 3, dtype=C128, device=DEV)
        box[:, (idx[:, 0] * N + idx[:, 1]) * N + idx[:, 2]] = u
        psi = torch.fft.ifftn(box.reshape(M, N, N, N), dim=(1, 2, 3)) * float(N ** 3)
        rho = (torch.from_numpy(f).to(DEV)[:, None, None, None] * psi.abs() ** 2).sum(0) / case["a"] ** 3
        return {"eig": e, "rho": rho}
    if fam == "rr":
        S, A, mu, T = _pencil(g, case["n"], case["m"])
        L = np.linalg.inv(np.linalg.cholesky(S.cpu().numpy()))
        h = L @ A.cpu().numpy() @ L.conj().T
        w, q = np.linalg.eigh(0.5 * (h + h.conj().T))
        theta = w[:case["m"]]
        c = L.conj().T @ q[:, :case["m"]]
        f = 1.0 / (1.0 + np.exp((theta - mu) / T))
        return {"theta": theta, "rho": np.ascontiguousarray(((c * f) @ c.conj().T).T)}
    if fam == "gemm_nn":
        a = _columns(g, case["k"], case["M"], prec).to(C128)
        b = _crandn(g, case["n"], case["k"]) / math.sqrt(case["k"])
        b = b.to(C64).to(C128) if prec == "c64" else b
        d = b @ a
        return d + _columns(g, case["n"], case["M"], prec).to(C128) if case["beta"] else d
    if fam == "gemm_cn":
        a = _columns(g, case["m"], case["K"], prec)
        b = _overlapping(g, a, case["n"], prec)
        return b.to(C128) @ a.to(C128).mH
    a = _columns(g, case["n"], case["K"], prec)
    return torch.triu(a @ a.mH)
