"""Tuned layout, 2 to 8 batch rows: which kernel takes a call on either side of the measured lines (148 SMs), and its result
there."""
import numpy as np
import pytest

from oracle import kmq_oracle as orc
from paper_2602_15563_b200 import kmq
from tests import gpu_util as gu
from tests.test_gpu_tcgen05 import random_layer

pytestmark = pytest.mark.gpu
TUNED = kmq.KMQ_LAYOUT_TUNED


@pytest.mark.parametrize("bits,N,K,M,kernel", [
    (1, 9600, 2048, 2, "tiled"), (1, 9600, 1536, 2, "multi"),          # a second wave: on 4 steps and more
    (1, 9472, 2048, 2, "multi"), (1, 9473, 2048, 4, "tiled"),          # four tiles per SM
    (1, 3072, 1536, 4, "tiled"), (1, 3072, 1024, 3, "multi"),          # odd and even numbers of steps
    (2, 2336, 8480, 4, "tiled"), (2, 3560, 8480, 2, "multi"),          # under and over one and a half tiles per SM
    (2, 1200, 16384, 5, "multi"), (2, 1200, 16112, 8, "tiled"),        # 64 and 63 steps
    (4, 9480, 2048, 3, "tiled"), (4, 9480, 1536, 3, "multi"),          # 16 and 12 steps of a second wave
    (4, 4160, 4096, 7, "multi"), (4, 4160, 4096, 6, "tiled"),
])
def test_kernel_on_either_side_of_a_line(bits, N, K, M, kernel):
    rng = np.random.default_rng(bits + N + K + M)
    idx, cb, x = random_layer(rng, N, K, bits, M)
    assert kmq.kmq_linear_variant(N, K, bits, M, TUNED).startswith(kernel)
    y_ref, s = orc.linear_f64(orc.pack_canonical(idx, bits), cb, x, K, bits)
    y = gu.gpu_linear(gu.gpu_pack(idx, bits, TUNED), cb, x, N, K, bits, TUNED)
    assert orc.check_linear(y, y_ref, s) <= 1.0


@pytest.mark.parametrize("bits,N,K,M,balanced", [
    (1, 12288, 4096, 8, False), (1, 16384, 12288, 8, True),
    (2, 9600, 4096, 8, False), (2, 9600, 6144, 8, True),
    (4, 8192, 12288, 3, False), (4, 8192, 16384, 3, True),
    (4, 6144, 4096, 8, False), (4, 6144, 8192, 8, True),
])
def test_balanced_form_on_either_side_of_its_line(bits, N, K, M, balanced):
    variant = kmq.kmq_linear_variant(N, K, bits, M, TUNED)
    assert variant.startswith("multi_balanced") == balanced, variant
