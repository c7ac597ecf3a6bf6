"""Complex64 tensor-core GEMMs (3xTF32) at the edges of their tiles: 128 left vectors, 32, 64 or 128
right columns, 8 reduction terms a stage, four stages in flight, one item per SM and round.

Against FP64 numpy.  Tolerance: the engine's stated 2e-6 of sum |a||b| for reductions of a few
hundred terms, and 1e-4 for the longest FP32 accumulation (4096 terms of one sign, each of whose
additions rounds by up to 2^-24 of the sum).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _rand(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("M", [1024, 1025, 1151, 128 * 152, 128 * 305 + 1])
@pytest.mark.parametrize("n,k", [(1, 1), (31, 7), (32, 8), (33, 9), (64, 31), (65, 33), (128, 40), (129, 64), (200, 5)])
def test_nn_tiles(M, n, k):
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(M + 1000 * n + k)
    A, B, C = _rand(rng, M, k), _rand(rng, k, n), _rand(rng, M, n)
    lg.set_gemm_mode(2)
    d = _dev(C.T)
    got = lg.gemm_nn(_dev(A.T), _dev(B.T), -1.5, 0.5, d, d).cpu().numpy().T     # in place
    lg.check_timeouts()
    A, B, C = A.astype(np.complex128), B.astype(np.complex128), C.astype(np.complex128)
    assert np.all(np.abs(got - (-1.5 * A @ B + 0.5 * C)) <= 2e-6 * (1.5 * np.abs(A) @ np.abs(B) + np.abs(C)))


@pytest.mark.parametrize("m,n", [(1, 1), (127, 32), (128, 33), (129, 64), (256, 65), (300, 129)])
@pytest.mark.parametrize("K", [1024, 1031, 4096, 9999])
def test_cn_tiles(m, n, K):
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(m + 1000 * n + K)
    A, B, C = _rand(rng, m, K), _rand(rng, n, K), _rand(rng, n, m)
    lg.set_gemm_mode(2)
    got = lg.gemm_cn(_dev(A), _dev(B), alpha=0.75, beta=-2.0, C=_dev(C)).cpu().numpy()
    lg.check_timeouts()
    A, B, C = A.astype(np.complex128), B.astype(np.complex128), C.astype(np.complex128)
    assert np.all(np.abs(got - (0.75 * B @ A.conj().T - 2.0 * C))
                  <= 2e-6 * (0.75 * np.abs(B) @ np.abs(A).T + 2 * np.abs(C)))


def test_cn_longest_accumulation():
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(3)
    A = np.abs(rng.standard_normal((1200, 57925))).astype(np.complex64)   # one sign: nothing cancels
    lg.set_gemm_mode(2)
    got = lg.gemm_cn(_dev(A), _dev(A)).cpu().numpy()
    want = A.real.astype(np.float64) @ A.real.astype(np.float64).T
    assert np.max(np.abs(got - want) / want) <= 1e-4
