"""The float32 dense preconditioner's quadrant products at the edges of their tiles (32, 64 and
128 outputs of a half side, 4-float pitches, odd sides whose middle entry is its own mirror),
against the float64 transform of the same map."""
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


# half sides one below, at and one above a tile's edge for the small (32), medium (64) and large
# (128) tiles; single rows and columns; sizes that select each tile (the last four: medium,
# medium, large, large)
SHAPES = [(1, 1), (1, 2), (2, 1), (5, 7), (62, 66), (63, 65), (64, 64), (65, 130), (126, 258),
          (255, 257), (1, 1000), (1000, 1), (1024, 1023), (1100, 2000), (1500, 1537), (4096, 2049)]


@pytest.mark.parametrize("H,W", SHAPES)
def test_quadrant_products_at_tile_edges(irls, H, W):
    """Within the float32 preconditioner's bound (2e-5 of the largest output), for an input at a
    16-byte boundary and one four bytes past it."""
    R = np.random.default_rng(H * 4099 + W).standard_normal((H, W)).astype(np.float32)
    ref = precond_reference_fft(R, 1e-2)
    scale = np.abs(ref).max()
    buf = torch.empty(H * W + 1, device="cuda")
    with irls.Plan(H, W, tau=1e-2, precision="fp32") as plan:
        assert plan.dct_form_name == "simt"
        out = []
        for off in (0, 1):
            x = buf[off:off + H * W].view(H, W)
            x.copy_(torch.as_tensor(R))
            out.append(irls.precond_laplacian(plan, x).cpu().numpy().astype(np.float64))
    assert np.array_equal(out[0], out[1])
    assert np.abs(out[0] - ref).max() <= 2e-5 * scale


def test_forms_of_one_plan_do_not_share_results(irls):
    """A plan's intermediates are shared by its forms: results do not depend on what ran before."""
    R = torch.as_tensor(np.random.default_rng(3).standard_normal((256, 512)).astype(np.float32)).cuda()
    with irls.Plan(256, 512, precision="fp32") as p:
        a = irls.precond_laplacian(p, R)
        p.set_opts(dct_form="fft")
        irls.precond_laplacian(p, R)
        p.set_opts(dct_form="auto")
        assert torch.equal(irls.precond_laplacian(p, R), a)
