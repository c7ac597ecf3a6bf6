"""Error of FP64-class tensor-core reductions against 64 bits, at shapes that could do with few splits.

A split's chunks of 64 terms are summed in double-FP32, the splits in FP64.  Measured before this test was
written, relative error of the whole product: 300 x 300 x 20000 3.9e-15 with at most 29 chunks a split, 4.5e-15
with 63; 200 x 90 x 60000 1.8e-15 and 2.0e-15; lower Gram 982 x 51039 9.3e-15 and 1.00e-14.  The limits lie
midway.
"""
import pytest

pytestmark = pytest.mark.gpu


def _columns(g, cols, rows):
    import torch
    d = 1.0 / (1.0 + 4.0 * torch.rand(rows, dtype=torch.float64, device="cuda", generator=g) ** 2)
    x = torch.complex(*(torch.randn(cols, rows, dtype=torch.float64, device="cuda", generator=g) for _ in range(2)))
    return x * (d * (0.5 ** 0.5 * 1.6 / rows ** 0.5))


@pytest.mark.parametrize("m,n,K,limit", [(300, 300, 20000, 4.2e-15), (200, 90, 60000, 1.9e-15), (982, 0, 51039, 9.65e-15)])
def test_error(m, n, K, limit):
    import torch
    import paper_0707_3405_gb300 as lg
    err = []
    for seed in range(3):
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        A = _columns(g, m, K)
        if n:       # columns that overlap with those of A
            B = 0.8 * A[m - n:] + 0.6 * _columns(g, n, K)
            got, want = lg.gemm_cn(A, B, tc=True), B @ A.mH
        else:
            got, want = torch.triu(lg.gram_lower(A, A, tc=True)), torch.triu(A @ A.mH)
        err.append((torch.linalg.vector_norm(got - want) / torch.linalg.vector_norm(want)).item())
    assert sum(err) / 3 <= limit, err
