"""FP64-class tensor-core GEMM: the work split over the SMs and the output forms.

Against numpy FP64 at sizes where the persistent schedule can go wrong (one item, fewer items than
SMs, a ragged last round, several slabs with a short last one), for every form of the output
(alpha, beta, accumulated slabs) and for operand scales outside the fast path.  Tolerance: the
engine's stated 2e-12 of sum |a||b|.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 2e-12


def _rand(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _close(got, want, a, b):
    assert np.all(np.abs(got - want) <= TOL * (np.abs(a) @ np.abs(b)))


# 64 rows = one left tile: 1, 151, 152, 153 and 305 tiles, and a ragged one
@pytest.mark.parametrize("M,n,k", [(64, 64, 64), (64 * 151, 64, 70), (64 * 152, 3, 64), (64 * 153, 64, 1),
                                   (64 * 152 + 37, 129, 200)])
@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-1.0, 1.0), (0.75, 0.0), (-1.0, 0.0)])
def test_nn_items_and_output_forms(M, n, k, alpha, beta):
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(M + n + k)
    A, B, C = _rand(rng, M, k), _rand(rng, k, n), _rand(rng, M, n)
    D = lg.gemm_nn(_dev(A.T), _dev(B.T), alpha, beta, _dev(C.T) if beta else None, tc=True).cpu().numpy().T
    want = alpha * (A @ B) + beta * C
    assert np.all(np.abs(D - want) <= TOL * (np.abs(A) @ np.abs(B) + np.abs(C)))
    lg.check_timeouts()


# (2048, 64): 244 chunks a slab, so 938 chunks run in four slabs, the last one short
@pytest.mark.parametrize("m,n,K", [(1, 1, 64), (128, 32, 64 * 5 + 1), (300, 70, 9001), (2048, 64, 60000)])
def test_cn_splits_and_slabs(m, n, K):
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(m + n + K)
    A, B = _rand(rng, m, K), _rand(rng, n, K)
    C = lg.gemm_cn(_dev(A), _dev(B), tc=True).cpu().numpy()
    _close(C, B @ A.conj().T, B, A.T)
    lg.check_timeouts()


@pytest.mark.parametrize("n", [1, 127, 129, 385, 700])
def test_lower_gram_tiles(n):
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(n)
    A = _rand(rng, n, 2000)
    C = lg.gram_lower(_dev(A), _dev(A), tc=True).cpu().numpy().T
    want = A.conj() @ A.T
    low = np.tril(np.ones((n, n), bool))
    assert np.all(np.abs(C - want)[low] <= TOL * (np.abs(A) @ np.abs(A.T))[low])
    lg.check_timeouts()


# columns of very different scale: 2^-55 x 2^-55 is below the normal range of a level's unit, 2^60 x
# 2^60 above it
@pytest.mark.parametrize("ea,eb", [(-55, -55), (60, 60), (-60, 60), (0, 0)])
def test_scales(ea, eb):
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(5)
    sa, sb = np.ones(130), np.ones(40)
    sa[1::2], sb[::3] = 2.0 ** ea, 2.0 ** eb
    A, B = _rand(rng, 130, 700) * sa[:, None], _rand(rng, 40, 700) * sb[:, None]
    C = lg.gemm_cn(_dev(A), _dev(B), tc=True).cpu().numpy()
    _close(C, B @ A.conj().T, B, A.T)
