"""Eigen-decompositions of nearly decoupled matrices: columns whose |x|^2 leaves the range of the arithmetic.

Every off-diagonal entry, or those between two halves, scaled down to where squares underflow (FP32, also in
pairs: 1e-19 to 1e-23; FP64: 1e-155 to 1e-162), in one cluster (n = 90) and in rows dealt to the SMs (200).
Tolerances as at scale 1: FP64 1e-12, double-FP32 n 2^-44, FP32 n 2^-20.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SCALES = [1.0, 1e-15, 1e-18, 1e-19, 1e-20, 1e-22, 1e-25, 1e-40]


def _herm(rng, n):
    a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    return a + a.conj().T


def _matrix(n, scale, kind):
    rng = np.random.default_rng(n)
    A = _herm(rng, n)
    if kind == "all":
        d = np.diag(A.diagonal().real)
        return d + scale * (A - d)
    h = n // 2
    A[h:, :h] *= scale
    A[:h, h:] *= scale
    return A


def _dev(x):
    import torch
    return torch.tensor(np.ascontiguousarray(x.T), device="cuda")


def _check(A, w, V, tol):
    nrm = np.abs(A).sum(1).max()
    assert np.isfinite(w).all() and np.isfinite(V).all()
    assert np.abs(w - np.linalg.eigvalsh(A)[:len(w)]).max() < tol * nrm
    assert np.abs(A @ V - V * w[None, :]).max() < 10 * tol * nrm
    assert np.abs(V.conj().T @ V - np.eye(len(w))).max() < tol


@pytest.mark.parametrize("kind", ["all", "between"])
@pytest.mark.parametrize("scale", SCALES)
@pytest.mark.parametrize("n", [90, 200])
def test_ritz_double_fp32(n, scale, kind):
    import paper_0707_3405_gb300 as lg
    A = _matrix(n, scale, kind)
    th, C, nd = lg.rayleigh_ritz(_dev(np.eye(n, dtype=complex)), _dev(A), n // 2, df32=True)
    assert int(nd.item()) == 0
    _check(A, th.cpu().numpy(), C.cpu().numpy().T, n * 2.0 ** -44)
    lg.check_timeouts()


@pytest.mark.parametrize("kind", ["all", "between"])
@pytest.mark.parametrize("scale", [1.0, 1e-20, 1e-155, 1e-160, 1e-163, 1e-200])
@pytest.mark.parametrize("n", [90, 200])
def test_heev_fp64(n, scale, kind):
    import paper_0707_3405_gb300 as lg
    A = _matrix(n, scale, kind)
    w, V = lg.heev(_dev(A))
    _check(A, w.cpu().numpy(), V.cpu().numpy().T, 1e-12)
    lg.check_timeouts()


@pytest.mark.parametrize("kind", ["all", "between"])
@pytest.mark.parametrize("scale", [1.0, 1e-15, 1e-20, 1e-25])
@pytest.mark.parametrize("n", [90, 200])
def test_ritz_fp32(n, scale, kind):
    import paper_0707_3405_gb300 as lg
    A = _matrix(n, scale, kind).astype(np.complex64)
    th, C, nd = lg.rayleigh_ritz32(_dev(np.eye(n, dtype=np.complex64)), _dev(A), n // 2)
    assert int(nd.item()) == 0
    _check(A.astype(complex), th.cpu().numpy().astype(float), C.cpu().numpy().T.astype(complex), n * 2.0 ** -20)
    lg.check_timeouts()

