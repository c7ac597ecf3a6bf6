"""FP64-class tensor-core products of few stages, back to back: a CTA leaves only when the last arrivals on its
barriers are in (its shared memory and TMEM go to the next launch's CTA at once)."""
import pytest

pytestmark = pytest.mark.gpu


def test_short_products_back_to_back():
    import torch
    import paper_0707_3405_gb300 as lg
    g = torch.Generator(device="cuda")
    g.manual_seed(0)
    ops = []
    for m, n, K in [(1, 1, 1), (130, 40, 64), (64, 33, 65), (300, 100, 200), (7, 5, 1000)]:
        A, B = (torch.randn(r, K, dtype=torch.complex128, device="cuda", generator=g) for r in (m, n))
        T = torch.randn(n, m, dtype=torch.complex128, device="cuda", generator=g)
        ops += [lambda A=A, B=B: lg.gemm_cn(A, B, tc=True), lambda A=A, T=T: lg.gemm_nn(A, T, tc=True)]
    first = [f() for f in ops]
    for _ in range(100):
        again = [f() for f in ops]
    lg.check_timeouts()
    for a, b in zip(first, again):
        assert torch.equal(a, b)
