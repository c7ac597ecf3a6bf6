"""Eigenvectors of matrices with a decoupled diagonal entry that an eigenvalue meets to the last bit: the pivot
of the inverse iteration is then the coupling itself, whose inverse squared overflowed to a zero vector.

diag + scale x full Hermitian, with so many eigenvalues that some are met exactly, in the row form of the
tridiagonalisation and in the per-column one (from n = 1217).  FP64 tolerances of the other sizes.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-20, 1e-60, 1e-100, 1e-155, 1e-160, 1e-200])
@pytest.mark.parametrize("n", [1000, 1216, 1217])
def test_heev_fp64(n, scale):
    import torch
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    A = A + A.conj().T
    d = np.diag(A.diagonal().real)
    A = d + scale * (A - d)
    w, V = lg.heev(torch.tensor(np.ascontiguousarray(A.T), device="cuda"))
    w, V = w.cpu().numpy(), V.cpu().numpy().T
    nrm = np.abs(A).sum(1).max()
    assert np.abs(w - np.linalg.eigvalsh(A)).max() < 1e-12 * nrm
    assert np.abs(A @ V - V * w[None, :]).max() < 1e-11 * nrm
    assert np.abs(V.conj().T @ V - np.eye(n)).max() < 1e-12
    lg.check_timeouts()
