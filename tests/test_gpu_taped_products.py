"""Recorded float32 solves run full-size preconditioner products, plain ones quadrants: the same
image, at the edges of both forms' tiles, on one plan in turn."""
import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def irls():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2401_09961_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("H,W", [(1, 40), (65, 64), (127, 130), (128, 128), (129, 257)])
def test_recorded_solve_equals_plain(irls, H, W):
    """Within 1e-3 rad, the bar between converged float32 solves; bit for bit between repeats."""
    from paper_2401_09961_gb300.autograd import unwrap_backward, unwrap_record

    d = synthetic.config_2048(seed=H + W, H=H, W=W)
    X = torch.as_tensor(d["X"], dtype=torch.float32).cuda()
    C = torch.as_tensor(d["coherence"], dtype=torch.float32).cuda()
    with irls.Plan(H, W, precision="fp32", tau=1e-2, delta=1e-3, outer_iters=2, cg_tol=1e-8,
                   cg_max_iter=1000) as p:
        U0 = p.unwrap(X, C)[0].clone()
        U1, tape, _ = unwrap_record(p, X, C)
        U1 = U1.clone()
        g1 = unwrap_backward(tape, torch.sin(U1))[0].clone()
        tape.free()
        U2 = p.unwrap(X, C)[0].clone()
        U3, tape, _ = unwrap_record(p, X, C)
        g3 = unwrap_backward(tape, torch.sin(U3))[0].clone()
        tape.free()
    assert torch.equal(U0, U2) and torch.equal(U1, U3) and torch.equal(g1, g3)
    assert float((U0 - U1).abs().max()) <= 1e-3
    assert bool(torch.isfinite(g1).all())
