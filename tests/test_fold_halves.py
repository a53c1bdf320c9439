"""Halved tiles of the folded launch's work list: the flag the kernel reads (it selects the operand
maps, the instruction's width and the epilogue) is exported for every stage and agrees with the
tiles, on the host."""
import numpy as np
import pytest

from test_fold_schedule import B, F, col, schedule  # noqa: F401

STAGE, HALF, WIDTH = "stage", "half", "width"


def check_halves(rec):
    half, stage = col(rec, HALF), col(rec, STAGE)
    assert set(np.unique(half)) <= {0, 1, 2}
    assert (stage[half == 1] == 3).all() and (stage[half == 2] == 2).all()
    two = col(rec, "dual") == 1
    assert ((half != 0) == (two & (col(rec, WIDTH) == 128))).all()
    # halves lie next to each other and share their whole tile
    at = np.where(half != 0)[0]
    assert len(at) % 2 == 0
    for i, j in zip(at[::2], at[1::2]):
        a, b = rec[i], rec[j]
        assert j == i + 1 and (a[[F["prob"], F["local"], F["m0"]]] ==
                               b[[F["prob"], F["local"], F["m0"]]]).all()
        assert a[F["n0"]] % 256 == 0 and b[F["n0"]] == a[F["n0"]] + 128
    # a stage's tiles are halved all together
    s2 = half[stage == 2]
    assert (s2 == s2[0]).all()


@pytest.mark.parametrize("shape", [(256, 256), (511, 769), (1024, 1024), (2047, 1999), (4096, 4096)])
@pytest.mark.parametrize("pairs", [1, 16, 76])
def test_flags_agree_with_the_tiles(B, shape, pairs):  # noqa: F811
    rec, _, _ = schedule(B, [shape], pairs)
    check_halves(rec)
    n2 = len(np.unique(rec[col(rec, STAGE) == 2][:, [F["prob"], F["local"]]], axis=0))
    assert (col(rec, HALF) == 2).any() == (2 * n2 <= pairs)


def test_planted_mistakes(B):  # noqa: F811
    rec, _, _ = schedule(B, [(1024, 1024)], 76)
    i = int(np.where(col(rec, HALF) == 2)[0][1])
    for field, value in ((HALF, 0), (HALF, 1), (WIDTH, 256)):
        r = rec.copy()
        r[i, F[field]] = value
        with pytest.raises(AssertionError):
            check_halves(r)
