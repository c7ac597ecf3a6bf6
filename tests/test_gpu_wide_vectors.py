"""Eigen-decompositions with all vectors where eight of them no longer fit the shared memory of the
back-transformation's block (n = 1752 in 16-byte entries)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1752, 1753, 2304])
@pytest.mark.parametrize("prec", ["fp64", "df32"])
def test_all_vectors(n, prec):
    import torch
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(n)
    a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    A = torch.tensor(a + a.conj().T, device="cuda")
    if prec == "fp64":
        w, V = lg.heev(A.T.contiguous())
        tol = 1e-12
    else:
        w, V, nd = lg.rayleigh_ritz(torch.eye(n, dtype=A.dtype, device="cuda"), A.T.contiguous(), n, df32=True)
        assert int(nd.item()) == 0
        tol = n * 2.0 ** -44
    V = V.T
    nrm = A.abs().sum(1).max()
    assert (w - torch.linalg.eigvalsh(A)).abs().max() < tol * nrm
    assert (A @ V - V * w[None, :]).abs().max() < 10 * tol * nrm
    assert (V.mH @ V - torch.eye(n, dtype=A.dtype, device="cuda")).abs().max() < tol
    lg.check_timeouts()
