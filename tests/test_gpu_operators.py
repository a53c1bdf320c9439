"""Single operators on the caller's own arrays: ragged strips, arrays at any alignment, outputs in
an input's place; the circular offset to FP64 accuracy over its branches."""
import ctypes

import numpy as np
import pytest

from oracle import irls as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def irls():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2401_09961_gb300 as m
    m.lib()
    return m


def at(a, off):
    """a on the GPU, starting `off` floats past a 16-byte boundary."""
    t = torch.empty(a.size + 4, device="cuda")[off:off + a.size].view(a.shape)
    return t.copy_(torch.as_tensor(a))


# a strip's ends: one row, one block of columns and a lane more, several strips with a short last
@pytest.mark.parametrize("H,W", [(1, 1), (1, 33), (33, 1), (2, 129), (700, 128), (1000, 1025)])
@pytest.mark.parametrize("off", [0, 1])
def test_apply_A_strips(irls, H, W, off):
    """Within the bound of the oracle comparison at other sizes (2e-6 of the largest + 1e-5)."""
    g = np.random.default_rng(H * 31 + W)
    f = lambda *s: g.standard_normal(s).astype(np.float32)  # noqa: E731
    U, Vv, Vh = f(H, W), f(H - 1, W), f(H, W - 1)
    Dv, Dh = (g.uniform(0, 1e3, s).astype(np.float32) for s in ((H - 1, W), (H, W - 1)))
    with irls.Plan(H, W, tau=1e-2) as p:
        q = irls.apply_A(p, *(at(a, off) for a in (U, Vv, Vh, Dv, Dh)))
    ref = O.apply_A(tuple(a.astype(np.float64) for a in (U, Vv, Vh)), Dv.astype(np.float64),
                    Dh.astype(np.float64), 1e-2)
    for a, b in zip(q, ref):
        if b.size:
            assert np.abs(a.cpu().numpy() - b).max() <= 2e-6 * np.abs(b).max() + 1e-5


def test_apply_A_in_place(irls):
    """Outputs written over the inputs: as into arrays of their own, bit for bit, and a later solve
    on the plan is unaffected."""
    H, W = 70, 93
    g = torch.Generator(device="cuda").manual_seed(1)
    r = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    U, Vv, Vh, Dv, Dh = r(H, W), r(H - 1, W), r(H, W - 1), r(H - 1, W).abs(), r(H, W - 1).abs()
    X = r(H, W)
    with irls.Plan(H, W, delta=1e-3, outer_iters=2) as p:
        U0, _ = p.unwrap(X)
        want = irls.apply_A(p, U, Vv, Vh, Dv, Dh)
        P = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
        rc = irls.lib().irls_apply_A(p.handle, P(U), P(Vv), P(Vh), P(Dv), P(Dh), P(U), P(Vv), P(Vh),
                                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        for a, b in zip((U, Vv, Vh), want):
            assert torch.equal(a, b)
        U1, _ = p.unwrap(X)
    assert torch.equal(U0, U1)


@pytest.mark.parametrize("prec,form", [("fp32", "auto"), ("bf16x3", "folded"), ("bf16x3", "direct"),
                                       ("fp32", "fft"), ("fp16", "folded")])
def test_precond_alignment_and_in_place(irls, prec, form):
    """Any alignment of the caller's array, and Z in R's place: the same bits."""
    R = np.random.default_rng(5).standard_normal((256, 512)).astype(np.float32)
    with irls.Plan(256, 512, precision=prec, dct_form=form) as p:
        Z = irls.precond_laplacian(p, at(R, 0))
        assert torch.equal(irls.precond_laplacian(p, at(R, 1)), Z)
        x = at(R, 0)
        P = ctypes.c_void_p(x.data_ptr())
        assert irls.lib().irls_precond_laplacian(
            p.handle, P, P, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
        assert torch.equal(x, Z)


@pytest.mark.parametrize("n,scale,off", [((1, 3), 1.0, 0), ((37, 53), 300.0, 1), ((700, 901), 3.0, 0),
                                         ((64, 65), 1e5, 0), ((1500, 1501), 8000.0, 1)])
def test_circular_offset_accuracy(irls, n, scale, off):
    """c and the best shift against FP64 numpy sums, over small and large phases (past 8192 rad the
    FP64 branch): sums of n terms of at most 1, each within 1e-15, so the direction of a sum of
    length L is within n 1e-15 / L (and FP64 atan2 rounding)."""
    g = np.random.default_rng(int(scale) + n[0])
    X = g.uniform(-np.pi, np.pi, n).astype(np.float32)
    U = (X + 2 * np.pi * np.rint(scale * g.standard_normal(n)) + 1.1 +
         0.3 * g.standard_normal(n)).astype(np.float32)
    d = U.astype(np.float64) - X.astype(np.float64)
    S, C = np.sin(d).sum(), np.cos(d).sum()
    with irls.Plan(*n) as p:
        _, K, c = irls.round_congruent(p, at(U, off), at(X, off))
        E, alpha, rms = irls.best_shift_error(p, at(U, off), at(X, off))
    assert abs(c - np.arctan2(S, C)) <= 1e-15 * d.size / np.hypot(S, C) + 1e-15 * 4
    assert np.array_equal(K.cpu().numpy(), O.round_congruent(U, X, c=c)[1])
    a = -d.mean()
    assert abs(alpha - a) <= 1e-14 * np.abs(d).mean() + 1e-15
    assert abs(rms - np.sqrt(np.mean((-d - a) ** 2))) <= 1e-13 * rms
