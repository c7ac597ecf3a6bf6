"""Rayleigh-Ritz steps at the block edges of the Cholesky factorisation and of the doubling inverse
(blocks of 32, pairs of 32, 64, 128 ..., the last one ragged), with dependent columns inside blocks,
and double-FP32 products of operands outside the middle of the FP32 range.

Tolerances: n 2^-44 of the norms for double-FP32 (2^-47 per operation), n 2^-48 for FP64.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _c(rng, *s):
    return rng.standard_normal(s) + 1j * rng.standard_normal(s)


@pytest.mark.parametrize("df32", [True, False])
@pytest.mark.parametrize("n,dep", [(1, ()), (31, ()), (32, (5,)), (33, (32,)), (65, (31, 32, 64)), (97, (10, 40, 70)),
                                   (161, (0,)), (224, (100, 223)), (300, (33, 34, 35, 290))])
def test_pencil_with_dropped_columns(n, dep, df32):
    import torch
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(n)
    dep = [d for d in dep if d > 0]
    Z = _c(rng, n + 40, n)
    for d in dep:
        Z[:, d] = Z[:, :d] @ _c(rng, d)        # dependent on the earlier columns
    Z /= np.linalg.norm(Z, axis=0)
    h = np.linspace(-1, 5, n + 40)
    S, A = Z.conj().T @ Z, Z.conj().T @ (h[:, None] * Z)
    m = max(1, (n - len(dep)) // 2)
    th, C, nd = lg.rayleigh_ritz(torch.tensor(S.T.copy(), device="cuda"), torch.tensor(A.T.copy(), device="cuda"), m,
                                 drop_tol=1e-9, df32=df32)
    assert int(nd.item()) == len(dep)
    th, C = th.cpu().numpy(), C.cpu().numpy().T
    tol = n * 2.0 ** (-44 if df32 else -48) * np.linalg.cond(np.delete(S, dep, 1)[[i for i in range(n) if i not in dep]])
    assert np.abs(C.conj().T @ S @ C - np.eye(m)).max() < tol
    R = Z @ C
    assert np.abs(R.conj().T @ (h[:, None] * R) - np.diag(th)).max() < 5 * tol


@pytest.mark.parametrize("ea,eb", [(0, 0), (-30, 30), (-70, 70), (100, -90)])
def test_double_fp32_products_over_the_range(ea, eb):
    import torch
    import paper_0707_3405_gb300 as lg
    rng = np.random.default_rng(7)
    A, B = _c(rng, 40, 300) * 2.0 ** ea, _c(rng, 30, 300) * 2.0 ** eb
    B[3] = 0.0
    C = lg.gemm_cn(torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda"), df32=True).cpu().numpy()
    # a pair holds 48 bits while its low part is a normal number: |x| above about 2^-78
    tol = 2e-12 if min(ea, eb) > -70 else 2.0 ** -30
    assert np.all(np.abs(C - B @ A.conj().T) <= tol * (np.abs(B) @ np.abs(A).T))
