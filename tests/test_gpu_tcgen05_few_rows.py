"""Up to 8 batch rows on the tcgen05 kernel: which calls go there on either side of the measured lines (148 SMs), and their
results; row lengths that leave CTAs of a cluster one stage or none at the end."""
import numpy as np
import pytest
import torch

from oracle import kmq_oracle as orc
from paper_2602_15563_b200 import kmq
from tests import gpu_util as gu
from tests.test_gpu_sum_error import layer
from tests.test_gpu_tcgen05 import random_layer

pytestmark = pytest.mark.gpu
TUNED = kmq.KMQ_LAYOUT_TUNED


@pytest.mark.parametrize("bits,N,K,M,tcgen05", [
    (4, 12033, 5640, 1, True), (4, 12033, 5568, 1, False), (4, 12032, 5640, 1, False),    # 2^26 weights; 95 and 94 blocks
    (4, 7041, 9536, 2, True), (4, 9473, 9536, 1, False), (4, 19000, 3600, 1, False),      # 56 and 75 blocks; a second wave
    (4, 5120, 13112, 1, True), (4, 5121, 13112, 1, False),
    (4, 10370, 4096, 3, True), (4, 10368, 4096, 3, False), (4, 10370, 4088, 5, False),    # 82 and 81 blocks
    (4, 12033, 2048, 8, True), (4, 12032, 2048, 8, False), (4, 12033, 2040, 4, False),
    (4, 6660, 6144, 5, True), (4, 6660, 6136, 5, False), (4, 6660, 4096, 6, True),
    (4, 5100, 3080, 4, True), (4, 5100, 3072, 8, True), (4, 5100, 3064, 8, False),
    (4, 900, 8192, 3, True), (4, 900, 6144, 7, True), (4, 896, 20480, 8, False), (4, 900, 6136, 6, False),
    (2, 14081, 4784, 6, True), (2, 14080, 4784, 6, False), (2, 14081, 4752, 8, False), (2, 14081, 4784, 5, False),
    (1, 16384, 8192, 8, False),
])
def test_few_rows_on_either_side_of_a_line(bits, N, K, M, tcgen05):
    assert kmq.kmq_linear_variant(N, K, bits, M, TUNED).startswith("tcgen05") == tcgen05
    if not tcgen05:
        return
    assert kmq.kmq_workspace_bytes(N, K, bits, M, TUNED) == 0
    rng = np.random.default_rng(bits + N + K + M)
    idx, cb, x = random_layer(rng, N, K, bits, M)
    y = gu.gpu_linear(gu.gpu_pack(idx, bits, TUNED), cb, x, N, K, bits, TUNED)
    rows = np.unique(np.concatenate([np.arange(0, N, 37), np.arange(N - 5, N)]))
    y_ref, s = orc.linear_f64(orc.pack_canonical(idx[rows], bits), cb[rows], x, K, bits)
    assert orc.check_linear(y[:, rows], y_ref, s) <= 1.0
    assert kmq.kmq_device_error_flags() == 0


@pytest.mark.parametrize("bits,N,K,M", [(4, 8192, 8192, 1), (4, 12033, 5640, 2), (4, 4312, 9216, 3), (4, 8259, 13696, 3),
                                        (4, 900, 28672, 8), (4, 5120, 28672, 1), (4, 4378, 21344, 5), (4, 12033, 2048, 8),
                                        (2, 16384, 8192, 8)])
def test_share_of_results_that_are_not_the_rounded_exact_ones(bits, N, K, M):
    """The bound of 9 to 16 batch rows, which run in the same form (8 accumulators): see tests/test_gpu_sum_error.py."""
    packed, cb, x, exact = layer(bits, N, K, M)
    assert kmq.kmq_linear_variant(N, K, bits, M, TUNED).startswith("tcgen05")
    y = torch.zeros(M, N, dtype=torch.bfloat16, device="cuda")
    kmq.kmq_linear(packed, cb, x, y, N, K, bits, M, None, 0, layout=TUNED)
    off = int((y != exact.float().to(torch.bfloat16)).sum())
    expected = (1.5 * 7.6e-6 * (K / 16) / 8 + 1e-4) * M * N
    assert off <= expected + 4 * expected ** 0.5     # few results: four standard deviations of their number
