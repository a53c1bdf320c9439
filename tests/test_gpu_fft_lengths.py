"""Every transform length of the fast-transform form, along rows and along columns: each has its
own sequence of stages (radix 16 with an 8, 4 or 2; radix 20 and 10), block shape and padding."""
import numpy as np
import pytest

from test_gpu_parity import precond_reference_fft

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def irls():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2401_09961_gb300 as m
    m.lib()
    return m


COLS = [64, 128, 256, 512, 1024, 2048, 4096, 8192, 2000, 4000, 8000]
ROWS = COLS + [16384, 16000]


@pytest.mark.parametrize("H,W", [(n, 128) for n in COLS] + [(64, n) for n in ROWS])
def test_each_length(irls, H, W):
    """Within 1e-5 (l2) and 2e-5 of the largest output: the bounds of the form's other tests."""
    R = np.random.default_rng(H + W).standard_normal((H, W)).astype(np.float32)
    ref = precond_reference_fft(R, 1e-2)
    with irls.Plan(H, W, tau=1e-2, precision="fp32", dct_form="fft") as p:
        Z = irls.precond_laplacian(p, torch.as_tensor(R).cuda()).cpu().numpy().astype(np.float64)
    assert np.linalg.norm(Z - ref) <= 1e-5 * np.linalg.norm(ref)
    assert np.abs(Z - ref).max() <= 2e-5 * np.abs(ref).max()
