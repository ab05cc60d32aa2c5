"""Short rows of many tiles on CTAs with as many warps as a row has steps (b = 1, 2): results against the oracle at ragged row
lengths and tile counts, and which kernel a call launches."""
import numpy as np
import pytest

from oracle import kmq_oracle as orc
from paper_2602_15563_b200 import kmq
from tests import gpu_util as gu
from tests.test_gpu_tcgen05 import random_layer

pytestmark = pytest.mark.gpu
TUNED = kmq.KMQ_LAYOUT_TUNED


@pytest.mark.parametrize("bits,N,K,M,warps", [
    (2, 9601, 64, 1, 4), (2, 12000, 1024, 1, 4), (2, 9601, 1040, 1, 8), (2, 3000, 1024, 1, 8), (2, 9480, 272, 2, 4),
    (2, 9495, 768, 3, 4), (2, 9000, 1024, 1, 8), (1, 12011, 32, 1, 4), (1, 9601, 2048, 1, 4), (1, 12000, 2080, 1, 6),
    (1, 1000, 2080, 1, 8), (1, 1003, 2592, 1, 6), (1, 1000, 3072, 2, 8), (1, 9600, 3072, 3, 6), (1, 1000, 3104, 1, 8),
])
def test_warps_by_steps(bits, N, K, M, warps):
    (name, grid, threads, _), = gu.linear_kernels(N, K, bits, M, TUNED)
    assert ("linear_tiled_short_kernel" in name) == (warps < 8) and "linear_tiled" in name
    assert threads == 32 * warps and grid[0] == -(-N // 16)
    rng = np.random.default_rng(bits + N + K + M)
    idx, cb, x = random_layer(rng, N, K, bits, M)
    y = gu.gpu_linear(gu.gpu_pack(idx, bits, TUNED), cb, x, N, K, bits, TUNED)
    y_ref, s = orc.linear_f64(orc.pack_canonical(idx, bits), cb, x, K, bits)
    assert orc.check_linear(y, y_ref, s) <= 1.0
