"""The bounded-wait path of the FP64-class tensor-core GEMMs, without hanging or faulting the GPU: with a
poll limit of zero the producer's first wait for a stage gives up at once, the device flag is raised, and the
wait is repeated with the full limit, so that the product is complete all the same."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,K", [(64, 32, 8192), (256, 128, 20000)])
def test_waits_run_out(m, n, K):
    import torch
    import paper_0707_3405_gb300 as lg
    g = torch.Generator(device="cuda")
    g.manual_seed(0)
    A, B = (torch.randn(r, K, dtype=torch.complex128, device="cuda", generator=g) for r in (m, n))
    T = torch.randn(n, m, dtype=torch.complex128, device="cuda", generator=g)
    calls = [lambda: lg.gemm_cn(A, B, tc=True), lambda: lg.gemm_nn(A, T, tc=True)]
    want = [f() for f in calls]
    lg.check_timeouts()
    for f, w in zip(calls, want):
        lg.set_spin_limit(0)
        try:
            late = f()
            with pytest.raises(lg.LobpcgError) as e:
                lg.check_timeouts()
        finally:
            lg.set_spin_limit(-1)
        assert e.value.code == lg.ERR_TIMEOUT
        lg.check_timeouts()                       # the flag was read and cleared
        assert torch.equal(late, w)
        assert torch.equal(f(), w)
        lg.check_timeouts()
