"""Tuned layout, small batches: K shared by a cluster of 2, 4 or 8 CTAs per tile (few tiles, long rows), ragged tiles and
row lengths."""
import numpy as np
import pytest

from oracle import kmq_oracle as orc
from paper_2602_15563_b200 import kmq
from tests import gpu_util as gu
from tests.test_gpu_tcgen05 import random_layer

pytestmark = pytest.mark.gpu
TUNED = kmq.KMQ_LAYOUT_TUNED


@pytest.mark.parametrize("bits", (1, 2, 4))
@pytest.mark.parametrize("N,K,M", [(1, 28672, 1), (100, 20000, 2), (250, 28640, 1), (500, 16416, 1), (590, 16352, 4),
                                   (1030, 12288, 1), (3070, 8224, 1), (700, 20000, 8)])
def test_rows_shared_by_a_cluster(bits, N, K, M):
    rng = np.random.default_rng(bits + N + K + M)
    idx, cb, x = random_layer(rng, N, K, bits, M)
    y_ref, s = orc.linear_f64(orc.pack_canonical(idx, bits), cb, x, K, bits)
    y = gu.gpu_linear(gu.gpu_pack(idx, bits, TUNED), cb, x, N, K, bits, TUNED)
    ratio = orc.check_linear(y, y_ref, s)
    assert ratio <= 1.0, f"error/tolerance = {ratio} [{kmq.kmq_linear_variant(N, K, bits, M, TUNED)}]"


@pytest.mark.parametrize("bits,N,K,kernel", [(1, 1000, 4096, "tiled"), (1, 1000, 20000, "multi"), (2, 4090, 9216, "multi"),
                                             (2, 3000, 16384, "tiled"), (4, 4790, 4096, "multi"), (4, 4000, 4104, "tiled")])
@pytest.mark.parametrize("M", (3, 4))
def test_which_kernel_takes_three_and_four_rows(bits, N, K, kernel, M):
    rng = np.random.default_rng(bits + N + K + M)
    idx, cb, x = random_layer(rng, N, K, bits, M)
    assert kmq.kmq_linear_variant(N, K, bits, M, TUNED).startswith(kernel)
    y_ref, s = orc.linear_f64(orc.pack_canonical(idx, bits), cb, x, K, bits)
    y = gu.gpu_linear(gu.gpu_pack(idx, bits, TUNED), cb, x, N, K, bits, TUNED)
    assert orc.check_linear(y, y_ref, s) <= 1.0
