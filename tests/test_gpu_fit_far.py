"""The fit on rows with values far out and with many next to zero: buckets from 4 to 256 times the unit and the one beyond, as many
members of a bucket as are looked at, sorted or searched in different ways, boundaries among them."""
import numpy as np
import pytest

from tests.test_gpu_fit_zero import fitted_alike

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("iters", (1, 20))
@pytest.mark.parametrize("bits", (1, 2, 4, 8))
@pytest.mark.parametrize("K", (512, 1056, 4096, 16384))
def test_values_far_out(K, bits, iters):
    """Normal rows of which a share is 6, 20, 100 and 3000 times as large, powers of two and their neighbours among them."""
    rng = np.random.default_rng(K + bits)
    W = rng.standard_normal((5, K)) * 0.02
    for row, factor in zip(W, (6, 20, 100, 3000, 1)):
        row[rng.random(K) < 0.2] *= factor
    W = W.astype(np.float32)
    far = rng.random(K) < 0.3
    W[4, far] = np.copysign(np.float32(2.0) ** rng.integers(-4, 6, far.sum()), W[4, far]).astype(np.float32)
    near = far & (rng.random(K) < 0.6)
    W[4, near] = np.nextafter(W[4, near], np.where(rng.random(near.sum()) < 0.5, np.float32(0), np.float32(99)))
    fitted_alike(W, bits, iters)


@pytest.mark.parametrize("octaves", (3, 22))
@pytest.mark.parametrize("members", (32, 33, 64, 65, 66, 67, 255, 256, 257))
@pytest.mark.parametrize("far", (False, True))
def test_members_of_the_buckets_of_mixed_octaves(members, octaves, far):
    """`members` values of each sign next to zero or beyond the last limit, over 3 octaves or more than add up without rounding (20;
    over 40 the sums of a row no longer hold its small values); 700 others so that quantiles, and boundaries after them, fall
    among them."""
    rng = np.random.default_rng(members + octaves + far)
    rows = []
    for others in (700, 701, 702, 703):
        scale = (1e4, 2.0 ** rng.integers(0, octaves, 2 * members)) if far else (1e-6, 2.0 ** -rng.integers(0, octaves, 2 * members))
        mixed = scale[0] * (1 + rng.random(2 * members)) * scale[1] * np.where(np.arange(2 * members) % 2 == 0, 1, -1)
        plain = (0.5 + rng.random(others)) * np.where(rng.random(others) < 0.5, 1, -1)
        rows.append(rng.permutation(np.concatenate([mixed, plain])))
    K = min(row.size for row in rows)
    W = np.stack([row[:K] for row in rows]).astype(np.float32)
    for bits in (1, 2, 4):
        for iters in (1, 20):
            fitted_alike(W, bits, iters)


@pytest.mark.parametrize("members", (63, 64, 65, 200, 384, 385))
def test_crowded_buckets(members):
    """That many values of each sign within a thousandth of each other, in one bucket that is neither at zero nor the last."""
    rng = np.random.default_rng(members)
    K = 2048
    W = rng.standard_normal((4, K)) * 0.02
    crowd = 0.0301 * (1 + 1e-3 * rng.random((4, 2 * members)))
    W[:, :2 * members] = np.where(np.arange(2 * members) % 2 == 0, crowd, -crowd)
    for bits in (1, 2, 4):
        for iters in (1, 20):
            fitted_alike(rng.permuted(W, axis=1).astype(np.float32), bits, iters)
