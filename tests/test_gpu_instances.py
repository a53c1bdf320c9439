"""The batch's instance of the direction and update kernels and every instance a single-image plan
takes (fixed and run-time row counts, both CG ratios) round alike: bit-identical results."""
import numpy as np
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


def cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32)).cuda()


SHAPES = [(333, 513), (701, 1003), (300, 2600)]


# the defaults (small images: run-time rows) and every fixed row count of either kernel
@pytest.mark.parametrize("flexible", [0, 1])
@pytest.mark.parametrize("tiles", [(24, 32), (8, 16), (16, 8), (32, 24)])
def test_batch_equals_plan(irls, tiles, flexible):
    opts = dict(tau=1e-2, delta=1e-3, outer_iters=2, cg_tol=1e-6, cg_max_iter=60,
                precision="bf16x3", dct_form="direct", flexible_cg=flexible)
    data = [synthetic.config_2048(seed=950 + t, H=h, W=w) for t, (h, w) in enumerate(SHAPES)]
    with irls.Batch(SHAPES, **opts) as b:
        b.set_tiles(*tiles)
        Us, st = b.unwrap([cuda(d["X"]) for d in data], [cuda(d["coherence"]) for d in data])
    for t, (h, w) in enumerate(SHAPES):
        with irls.Plan(h, w, **opts) as p:
            p.set_tiles(*tiles)
            U, s1 = p.unwrap(cuda(data[t]["X"]), cuda(data[t]["coherence"]))
        assert torch.equal(Us[t], U), SHAPES[t]
        assert st[t]["rel_res"] == s1["rel_res"] and st[t]["l1_obj"] == s1["l1_obj"], SHAPES[t]
