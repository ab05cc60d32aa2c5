"""The row-major tensor-core kernel (canonical layout of any row length; block format) and the tuned-layout kernels on
row lengths that are no whole number of 16-byte chunks: ends of rows and tiles, every number of batch rows per operand,
both CTA sizes."""
import numpy as np
import pytest

from oracle import kmq_oracle as orc
from paper_2602_15563_b200 import kmq, synth
from tests import gpu_util as gu
from tests.test_gpu_block import run_all
from tests.test_gpu_tcgen05 import random_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", (kmq.KMQ_LAYOUT_CANONICAL, kmq.KMQ_LAYOUT_TUNED))
@pytest.mark.parametrize("bits", (1, 2, 4))
@pytest.mark.parametrize("N,words,M", [(1, 1, 1), (16, 3, 8), (17, 5, 9), (33, 17, 4), (70, 90, 2), (250, 33, 17),
                                       (2400, 41, 3), (40, 130, 40), (300, 29, 140)])
def test_row_lengths_of_odd_words(bits, N, words, M, layout):
    K = words * (32 // bits)
    rng = np.random.default_rng(bits * 1000 + N + words)
    idx, cb, x = random_layer(rng, N, K, bits, M)
    y_ref, s = orc.linear_f64(orc.pack_canonical(idx, bits), cb, x, K, bits)
    y = gu.gpu_linear(gu.gpu_pack(idx, bits, layout), cb, x, N, K, bits, layout)
    ratio = orc.check_linear(y, y_ref, s)
    assert ratio <= 1.0, f"error/tolerance = {ratio} [{kmq.kmq_linear_variant(N, K, bits, M, layout)}]"


@pytest.mark.parametrize("bits", (1, 2, 4, 8))
@pytest.mark.parametrize("N,K,M", [(1, 64, 1), (17, 64 * 7, 8), (40, 64 * 33, 9), (2400, 64 * 9, 16), (90, 64 * 20, 33)])
def test_block_format(bits, N, K, M):
    rng = np.random.default_rng(bits * 100 + N + M)
    Q = 1 << bits
    idx = rng.integers(0, Q, size=(N, K), dtype=np.uint8)
    scales = synth.f32_to_bf16_bits((rng.random((N, K // 64)) * 0.1 + 1e-3).astype(np.float32))
    cb = synth.f32_to_bf16_bits(np.sort(rng.standard_normal(Q)).astype(np.float32))
    x = synth.f32_to_bf16_bits(rng.standard_normal((M, K)).astype(np.float32))
    assert run_all(idx, scales, cb, x, bits, f"N={N} K={K} M={M}") <= 1.0
