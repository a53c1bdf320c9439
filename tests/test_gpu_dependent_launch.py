"""Dependent launches of the float32 CG kernels: runs on two streams from two threads at once, three
each, equal a run alone bit for bit."""
import threading

import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

OPTS = dict(tau=1e-2, delta=1e-3, outer_iters=3, cg_tol=1e-6, cg_max_iter=200)


@pytest.fixture(scope="module")
def irls():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2401_09961_gb300 as m
    m.lib()
    return m


def image(h, w, seed):
    d = synthetic.config_2048(seed=seed, H=h, W=w)
    return (torch.as_tensor(d["X"], dtype=torch.float32).cuda(),
            torch.as_tensor(d["coherence"], dtype=torch.float32).cuda())


@pytest.mark.parametrize("shapes,kw", [
    ([(1, 37), (64, 64)], dict(precision="fp32")),
    ([(257, 391), (300, 451)], dict(precision="fp32")),
    ([(512, 256), (256, 512)], dict(precision="fp32", dct_form="fft")),
    ([(512, 256), (256, 512)], dict(precision="fp32", dct_form="fft", system="schur"))])
def test_two_streams_equal_one(irls, shapes, kw):
    ims = [image(h, w, h + w) for h, w in shapes]
    alone, both = [], [None, None]
    for X, C in ims:
        with irls.Plan(*X.shape, **kw, **OPTS) as p:
            alone.append(p.unwrap(X, C)[0].clone())
    torch.cuda.synchronize()

    def run(i):
        X, C = ims[i]
        with torch.cuda.stream(torch.cuda.Stream()), irls.Plan(*X.shape, **kw, **OPTS) as p:
            both[i] = [p.unwrap(X, C)[0].clone() for _ in range(3)]
            torch.cuda.current_stream().synchronize()

    ts = [threading.Thread(target=run, args=(i,)) for i in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for i in range(2):
        assert both[i] is not None and all(torch.equal(u, alone[i]) for u in both[i])
