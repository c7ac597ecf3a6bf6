"""Eigen-decompositions at the sizes where the tridiagonalisation changes its form or its split: one
cluster up to n = 128, rows dealt to the SMs above (one row, then two, per block at 152 and 153; the
last size that fits their shared memory is below 1217), and the per-column kernels beyond.

Tolerances: the FP64 checks of the other sizes; double-FP32 with 2^-47 per operation, n 2^-44.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SIZES = [127, 128, 129, 152, 153, 305, 700, 1217]


def _herm(rng, n):
    a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    return a + a.conj().T


@pytest.mark.parametrize("n", SIZES)
def test_heev_fp64(n):
    import torch
    import paper_0707_3405_gb300 as lg
    A = _herm(np.random.default_rng(n), n)
    w, V = lg.heev(torch.tensor(A.T.copy(), device="cuda"))
    w, V = w.cpu().numpy(), V.cpu().numpy().T
    nrm = np.abs(A).sum(1).max()
    assert np.abs(w - np.linalg.eigvalsh(A)).max() < 1e-12 * nrm
    assert np.abs(A @ V - V * w[None, :]).max() < 1e-11 * nrm
    assert np.abs(V.conj().T @ V - np.eye(n)).max() < 1e-12
    lg.check_timeouts()


@pytest.mark.parametrize("n", SIZES)
def test_ritz_double_fp32(n):
    import torch
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(n)
    A = _herm(rng, n)
    S = np.eye(n) + 0.2 * _herm(rng, n) / (4.0 * np.sqrt(n))
    m = n // 2
    th, C, nd = lg.rayleigh_ritz(torch.tensor(S.T.copy(), device="cuda"), torch.tensor(A.T.copy(), device="cuda"), m,
                                 df32=True)
    th, C = th.cpu().numpy(), C.cpu().numpy().T
    nrm = np.abs(A).sum(1).max()
    assert int(nd.item()) == 0
    assert np.abs(A @ C - S @ C * th[None, :]).max() < n * 2.0 ** -44 * nrm
    assert np.abs(C.conj().T @ S @ C - np.eye(m)).max() < n * 2.0 ** -44
    lg.check_timeouts()


def test_diagonal_and_zero_columns():
    # reflectors of zero columns (tau = 0) in the row form
    import torch
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(3)
    A = np.diag(rng.standard_normal(200)).astype(complex)
    A[150:, 150:] = _herm(rng, 50)
    w, V = lg.heev(torch.tensor(A.T.copy(), device="cuda"))
    w, V = w.cpu().numpy(), V.cpu().numpy().T
    assert np.abs(w - np.linalg.eigvalsh(A)).max() < 1e-12 * np.abs(A).sum(1).max()
    assert np.abs(V.conj().T @ V - np.eye(200)).max() < 1e-12


@pytest.mark.parametrize("scale", [1.0, 1e14, 1e-14, 1e30, 1e-30])
def test_heev_scales(scale):
    # the multisection's FP32 and double-FP32 rounds in and out of their range
    import torch
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(9)
    A = _herm(rng, 90) * scale
    w, V = lg.heev(torch.tensor(A.T.copy(), device="cuda"))
    w, V = w.cpu().numpy(), V.cpu().numpy().T
    nrm = np.abs(A).sum(1).max()
    assert np.abs(w - np.linalg.eigvalsh(A)).max() < 1e-13 * nrm
    assert np.abs(V.conj().T @ V - np.eye(90)).max() < 1e-12


@pytest.mark.parametrize("n", [2, 3, 33, 90, 200])
@pytest.mark.parametrize("kind", ["wide", "near", "clusters", "equal", "blocks"])
def test_heev_spectra(kind, n):
    # inverse iteration at the edge of a cluster: neighbours 2e-5 |T| apart are solved alone (their vectors
    # are orthogonal to about eps / 2e-5, times 16), closer ones together
    import torch
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(n)
    if kind == "wide":
        lam = np.arange(n) - n / 3.0
    elif kind == "near":
        lam = np.where(np.arange(n) % 2 == 0, np.arange(n), np.arange(n) - 1 + 4e-5 * n)
    elif kind == "clusters":
        lam = np.floor(np.arange(n) / 5.0) + 1e-9 * np.arange(n)
    elif kind == "equal":
        lam = np.full(n, 0.75)
    else:
        lam = np.arange(n) * 1.0
    Q = np.linalg.qr(_herm(rng, n))[0] if kind != "blocks" else np.eye(n)
    A = (Q * lam) @ Q.conj().T
    A = (0.5 * (A + A.conj().T)).astype(complex)
    w, V = lg.heev(torch.tensor(A.T.copy(), device="cuda"))
    w, V = w.cpu().numpy(), V.cpu().numpy().T
    nrm = np.abs(A).sum(1).max()
    assert np.abs(w - np.linalg.eigvalsh(A)).max() < 1e-12 * nrm
    assert np.abs(A @ V - V * w[None, :]).max() < 1e-11 * nrm
    assert np.abs(V.conj().T @ V - np.eye(n)).max() < 16 * 2.0 ** -52 / 1e-5
