"""Double-FP32 products of FP64 numbers near the lower end of FP32.

A pair holds such a number to two roundings of at most half of 2^-149 each (hi, then lo).  The sum of |a||b| over
entries of size 1e-40 then carries a relative error of at most 2 x 2^-149 / 1e-40 x E|b| / (E|a| E|b|), with E|a| =
E|b| = 0.89 x sqrt(2): 2.3e-5.  (Numbers below 2^-138 taken as zero leave 3e-4.)
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [500, 2000])
def test_tiny_operand(K):
    import torch
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(K)
    A, B = (rng.standard_normal((n, K)) + 1j * rng.standard_normal((n, K)) for n in (64, 32))
    A = A * 1e-40
    got = lg.gemm_cn(torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda"), df32=True).cpu().numpy()
    assert np.max(np.abs(got - B @ A.conj().T) / (np.abs(B) @ np.abs(A).T)) <= 2.3e-5
