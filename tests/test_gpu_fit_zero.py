"""The fit's buckets at zero and at their limits: as many members next to zero as have their partial sums kept, one more, many
more; members of more octaves than can be added up without rounding; values on the limits of buckets, powers of two among them."""
import numpy as np
import pytest

from tests.test_gpu_quantize import check_fit

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("octaves", (3, 60))
@pytest.mark.parametrize("members", (1, 2, 31, 32, 33, 63, 64, 65, 200))
def test_members_next_to_zero(members, octaves):
    """`members` values of each sign far below the rest, so that a boundary of the symmetric row lies among them."""
    rng = np.random.default_rng(members + octaves)
    K = 4096
    W = rng.standard_normal((4, K)) * 0.02
    W = np.where(np.abs(W) < 1e-3, np.copysign(1e-3, W), W)
    tiny = 1e-5 * rng.random((4, 2 * members)) * 2.0 ** -rng.integers(0, octaves, (4, 2 * members))
    W[:, :members] = tiny[:, :members]
    W[:, members:2 * members] = -tiny[:, members:]
    W[3, :2 * members] = np.where(np.arange(2 * members) % 2 == 0, 0.0, -0.0)
    for bits in (1, 4):
        check_fit(rng.permuted(W, axis=1).astype(np.float32), bits)


@pytest.mark.parametrize("scale", (1.0, 2.0 ** -100, 2.0 ** 100))
@pytest.mark.parametrize("K", (1024, 4096, 32768))
def test_values_on_the_limits_of_buckets(K, scale):
    """Multiples of a power of two, up to 8 times the row's typical magnitude, with neighbours one step on either side."""
    rng = np.random.default_rng(K)
    steps = rng.integers(-4 * K, 4 * K + 1, K).astype(np.float32) / np.float32(K)
    W = np.stack([steps, np.nextafter(steps, np.float32(9)), np.nextafter(steps, np.float32(-9))])
    W *= np.abs(rng.standard_normal((3, K))).astype(np.float32) > 0.3
    check_fit((W * np.float32(scale)).astype(np.float32), 4)
