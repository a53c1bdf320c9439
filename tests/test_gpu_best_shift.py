"""Best shift against its definition in extended precision: an offset far larger than the errors,
values whose squares leave float32's range, and pixels that are not finite."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def irls():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2401_09961_gb300 as m
    m.lib()
    return m


def shift(irls, U, Xu):
    with irls.Plan(*U.shape) as p:
        E, alpha, rms = irls.best_shift_error(p, torch.as_tensor(U).cuda(), torch.as_tensor(Xu).cuda())
    return E.cpu().numpy(), alpha, rms


def wide(n, scale, offset, noise, seed):
    g = np.random.default_rng(seed)
    U = (scale * g.uniform(-1, 1, n)).astype(np.float32)
    return U, (U + np.float64(offset) + noise * g.standard_normal(n)).astype(np.float32)


# offset far above the errors (their second parts count), the other way round, squares above and
# below float32's range, sums of four above it
@pytest.mark.parametrize("n,scale,offset,noise", [
    ((601, 503), 500.0, 1000.0, 1e-3), ((64, 63), 30.0, 200.0, 1e-4), ((300, 301), 1.0, 1e-3, 3.0),
    ((64, 65), 1e20, 1e19, 1e21), ((33, 35), 1e38, 2e37, 1e37), ((64, 61), 1e-18, 1e-17, 1e-19),
    ((64, 61), 1e-12, 1e-11, 1e-16)])
def test_accuracy(irls, n, scale, offset, noise):
    """alpha within n FP64 roundings of the differences' mean magnitude; a square carries 46 bits
    and more (relative 2^-46 = 1.4e-14), rms half of that and its FP64 sums: 1e-13."""
    U, Xu = wide(n, scale, offset, noise, n[1])
    E, alpha, rms = shift(irls, U, Xu)
    d = Xu.astype(np.longdouble) - U.astype(np.longdouble)
    a = d.mean()
    assert abs(alpha - a) <= 1e-14 * np.abs(d).mean()
    ref = np.sqrt(((d - np.longdouble(alpha)) ** 2).mean())
    assert abs(rms - ref) <= 1e-13 * ref
    assert np.array_equal(E, (Xu - U) - np.float32(alpha))


def test_identical_images(irls):
    U, _ = wide((50, 51), 10.0, 0.0, 0.0, 3)
    E, alpha, rms = shift(irls, U, U)
    assert alpha == 0.0 and rms == 0.0 and not E.any()


# a pixel in a whole group of four, and in the last, shorter one
@pytest.mark.parametrize("where", [17, -1])
@pytest.mark.parametrize("u,x", [(0.0, np.inf), (0.0, -np.inf), (np.inf, 0.0), (np.inf, np.inf),
                                 (np.nan, 0.0)])
def test_not_finite(irls, where, u, x):
    U, Xu = wide((37, 41), 10.0, 5.0, 0.1, 9)
    U.flat[where], Xu.flat[where] = u, x
    E, alpha, rms = shift(irls, U, Xu)
    with np.errstate(invalid="ignore"):
        d = Xu.astype(np.float64) - U.astype(np.float64)
        a = d.mean()
        assert np.array_equal(alpha, a, equal_nan=True)
        assert np.array_equal(rms, np.sqrt(((d - a) ** 2).mean()), equal_nan=True)
        assert np.array_equal(E, (Xu - U) - np.float32(alpha), equal_nan=True)
