"""The live profiler over a CG run longer than the event pairs it holds: every launch is counted."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", ["fp32", "bf16x3"])
def test_long_run_counts(prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2401_09961_gb300 as irls
    X = torch.randn(256, 300, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    L = irls.lib()
    with irls.Plan(256, 300, precision=prec, tau=1e-2, delta=1e-3, outer_iters=2, cg_tol=0.0,
                   cg_max_iter=150) as p:
        U0, _ = p.unwrap(X)
        L.irls_plan_set_profiling(p.handle, 1)
        U1, st = p.unwrap(X)
        ms, n = (ctypes.c_double * 6)(), (ctypes.c_longlong * 6)()
        assert L.irls_plan_profile(p.handle, ms, n, 6) == 6
        L.irls_plan_set_profiling(p.handle, 0)
    assert torch.equal(U0, U1) and st["cg_iters"] == [150, 150]
    assert list(n[1:6]) == [2, 300, 300, 302, 2] and n[0] >= 1
    assert all(m > 0 for m in ms)
