"""The fit's buckets at zero and at their limits: as many members next to zero as have their partial sums kept, one more, many
more; members of more octaves than can be added up without rounding; values on the limits of buckets, powers of two among them;
boundaries of -0.0, which belong to the zeros of both signs."""
import numpy as np
import pytest

from tests.test_gpu_quantize import check_fit, gpu_fit

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


def masked_rows(K, share, seed):
    """Normal rows times a mask of zeros and ones: a zero of either sign for every weight that is masked out."""
    rng = np.random.default_rng(seed)
    return (rng.standard_normal((24, K)) * 0.02 * (rng.random((24, K)) >= share)).astype(np.float32)


def fitted_alike(W, bits, iters):
    """Against the oracle, and bit for bit the same once more after other rows have been in the same shared memory."""
    check_fit(W, bits, iters)
    first = gpu_fit(W, bits, iters)
    gpu_fit(np.flip(W, axis=0) * np.float32(3), bits, iters)
    for a, b in zip(first, gpu_fit(W, bits, iters)):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("iters", (1, 2, 20))
@pytest.mark.parametrize("bits", (1, 2, 4, 8))
@pytest.mark.parametrize("K", (32, 96, 160, 256, 544, 1024))
def test_rows_of_masked_weights(K, bits, iters):
    """Neighbouring start quantiles in the run of -0.0 make a boundary of -0.0: all zeros lie at or below it."""
    if K < 1 << bits:
        pytest.skip("fewer values than centroids")
    fitted_alike(np.concatenate([masked_rows(K, share, K + bits + int(100 * share)) for share in (0.1, 0.3, 0.5, 0.7)]), bits, iters)


@pytest.mark.parametrize("iters", (1, 3))
@pytest.mark.parametrize("members", (30, 31, 32, 33, 63, 64, 65))
def test_boundary_of_negative_zero(members, iters):
    """`members` of -0.0, as many and fewer of +0.0, and as many values below them that every place modulo 4 is a start."""
    rng = np.random.default_rng(members)
    rows = []
    for below in range(3 * members, 3 * members + 4):
        for positive in (members, 5):
            above = 8 * members - below - members - positive
            row = np.concatenate([-0.01 - rng.random(below), np.full(members, -0.0), np.zeros(positive), 0.01 + rng.random(above)])
            rows.append(rng.permutation(row))
    fitted_alike(np.stack(rows).astype(np.float32), 4, iters)
