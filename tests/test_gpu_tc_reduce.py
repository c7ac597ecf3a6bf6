"""Sum of the partial tiles of the complex64 reductions: alpha (sum) + beta C rounded once, and partial sums
that leave the FP32 range on the way."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _gemm_cn(A, B, **kw):
    import torch
    import paper_0707_3405_gb300 as lg
    lg.set_gemm_mode(2)
    kw = {k: torch.from_numpy(v).cuda() if isinstance(v, np.ndarray) else v for k, v in kw.items()}
    got = lg.gemm_cn(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), **kw).cpu().numpy()
    lg.check_timeouts()
    return got


@pytest.mark.parametrize("K", [1024, 5000, 57925])
def test_one_rounding(K):
    """Small integers: every partial sum is exact (below 2^24), so alpha (sum) + beta C in FP64, rounded to
    FP32, is the result (FP64's own rounding decides one entry in 2^28)."""
    rng = np.random.default_rng(K)
    A, B = (rng.integers(-3, 4, (40, K)) + 1j * rng.integers(-3, 4, (40, K)) for _ in range(2))
    C = (rng.standard_normal((40, 40)) + 1j * rng.standard_normal((40, 40))).astype(np.complex64) * 100
    al, be = np.float32(0.3), np.float32(-1.7)
    want = float(al) * (B @ A.conj().T) + float(be) * C.astype(complex)
    got = _gemm_cn(A.astype(np.complex64), B.astype(np.complex64), alpha=float(al), beta=float(be), C=C)
    assert np.array_equal(got, want.astype(np.complex64))


def test_range():
    """1e18 x 1e18: 256 terms of a chunk are finite, the sum of 512 is not, 512 more of the other sign bring
    it back to zero; 1e19 x 1e19 overflows in every chunk, to infinity."""
    A = np.full((8, 1024), 1e18, np.complex64)
    B = A.copy()
    B[:, 512:] *= -1
    assert np.array_equal(_gemm_cn(A, B), np.zeros((8, 8), np.complex64))
    got = _gemm_cn(A * np.float32(10), A * np.float32(10), alpha=-1.0)
    assert np.all(got.real == -np.inf) and not got.imag.any()
