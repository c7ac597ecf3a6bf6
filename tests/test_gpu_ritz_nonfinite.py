"""A pencil with an entry that is infinite or not a number has no finite Ritz values in the double-FP32 step,
wherever the entry is: the products with the triangular inverse skip its zeros, so it need not spread."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("at", [(0, 0), (-1, -1), (-1, 0), (-1, -2), (40, 39)])
@pytest.mark.parametrize("n", [45, 90, 200, 640])
def test_ritz_values(n, at, bad):
    import torch
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    A = A + A.conj().T
    A[at] = bad
    S = torch.eye(n, dtype=torch.complex128, device="cuda")
    theta, C, nd = lg.rayleigh_ritz(S, torch.tensor(np.ascontiguousarray(A.T), device="cuda"), n // 3, df32=True)
    assert not torch.isfinite(theta).any()
    assert not torch.isfinite(C.real).any()
