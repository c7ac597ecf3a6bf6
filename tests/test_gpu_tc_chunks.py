"""Complex64 reductions A^H B on the tensor cores: their FP32 chunks depend on the reduction length alone.

The tensor core truncates as it accumulates.  The Gram matrices S and A of one Rayleigh-Ritz step have
different shapes, and where A lost more than S (longer chunks) spurious Ritz values appeared; so an entry is the
same, to the bit, whatever block it is computed in, and chunks have at most 1024 terms.
"""
import pytest

pytestmark = pytest.mark.gpu


def _randn(rows, K, seed):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(rows, K, dtype=torch.complex64, device="cuda", generator=g)


@pytest.mark.parametrize("K", [1024, 4099, 57925, 113081])
def test_entries_do_not_depend_on_the_block(K):
    import torch
    import paper_0707_3405_gb300 as lg
    lg.set_gemm_mode(2)
    A, B = _randn(400, K, 1), _randn(300, K, 2)
    whole = lg.gemm_cn(A, B)
    for m, n in [(384, 256), (256, 256), (128, 128), (100, 70), (33, 40), (20, 20), (400, 64), (7, 300)]:
        assert torch.equal(lg.gemm_cn(A[:m].contiguous(), B[:n].contiguous()), whole[:n, :m]), (m, n)
    lg.check_timeouts()


def test_panels():
    """A product whose partial tiles exceed their scratch runs in panels of rows and columns."""
    import torch
    import paper_0707_3405_gb300 as lg
    lg.set_gemm_mode(2)
    A, B, C0 = _randn(1700, 113081, 3), _randn(300, 113081, 4), _randn(300, 1700, 5)
    got = lg.gemm_cn(A, B, alpha=0.5, beta=2.0, C=C0.clone())
    for i, j in [(0, 0), (1500, 0), (0, 150), (1500, 150)]:
        sub = lg.gemm_cn(A[i:i + 200].contiguous(), B[j:j + 150].contiguous(), alpha=0.5, beta=2.0,
                         C=C0[j:j + 150, i:i + 200].contiguous())
        assert torch.equal(sub, got[j:j + 150, i:i + 200]), (i, j)
    lg.check_timeouts()


@pytest.mark.parametrize("m,n", [(384, 256), (256, 256), (128, 128)])
@pytest.mark.parametrize("K", [113081, 155000])
def test_truncation(m, n, K):
    """Sums of one sign: a chunk of 1024 terms takes 3 x 256 MMAs, each of which truncates half a unit
    in the last place (at most 2^-23 of the sum so far, which is half the final one on average): the mean
    shortfall is at most 768 x 2^-25 = 2.3e-5."""
    import torch
    import paper_0707_3405_gb300 as lg
    lg.set_gemm_mode(2)
    A = _randn(m, K, 6).real.abs().to(torch.complex64)
    B = A[:n].contiguous()
    got = lg.gemm_cn(A, B).real.double()
    want = B.real.double() @ A.real.double().T
    assert abs(((got - want) / want).mean().item()) <= 768 * 2.0 ** -25


def test_very_long_reduction():
    """More terms than 4 x 152 chunks of 4096."""
    import paper_0707_3405_gb300 as lg
    lg.set_gemm_mode(2)
    A = _randn(3, 2_600_001, 7)
    got = lg.gemm_cn(A, A)
    lg.check_timeouts()
    a = A.to(got.dtype).cdouble()
    want = a @ a.mH
    assert ((got - want.to(got.dtype)).abs().max() / want.abs().max()).item() <= 768 * 2.0 ** -24
