"""The medium and large tiles of the float32 dense preconditioner one below, at and one above their
edges, against the float64 transform of the same map.  Which tile a size takes is restated here from
the rule's measured costs, so that the sizes stay where they are meant to be."""
import pytest

from test_gpu_dense_f32 import irls, test_quadrant_products_at_tile_edges as check  # noqa: F401

CASES = [  # half sides
    (1022, 1024, 64),    # 511 x 512
    (1023, 1025, 64),    # 512 x 513
    (1150, 1151, 64),    # 575 x 576
    (1500, 1537, 64),    # 750 x 769
    (1534, 1535, 128),   # 767 x 768
    (1530, 1536, 128),   # 765 x 768
    (4096, 2049, 128),   # 2048 x 1025
]


def tile(m, n, sms=152):
    """128, 64 or 32: the least busy-SM time, in large tiles."""
    def waves(b):
        return -(-(-(-m // b) * -(-n // b) * 4) // sms)
    cost = {128: waves(128), 64: waves(64) / 4 / 0.88, 32: waves(32) / 16 / 0.62}
    return min((128, 64, 32), key=cost.get)


@pytest.mark.parametrize("H,W,want", CASES)
def test_the_rule_takes_the_tile(H, W, want):
    h, w = (H + 1) // 2, (W + 1) // 2
    assert tile(w, h) == want and tile(h, w) == want


@pytest.mark.gpu
@pytest.mark.parametrize("H,W", [c[:2] for c in CASES])
def test_products_at_the_edges(irls, H, W):  # noqa: F811
    check(irls, H, W)
