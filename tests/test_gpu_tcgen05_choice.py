"""Tuned layout, 9 batch rows and more: which kernel takes a call on either side of the measured lines (148 SMs), and its
result there; the edges of the tcgen05 kernel's rings, clusters and batch widths."""
import numpy as np
import pytest
import torch

from oracle import kmq_oracle as orc
from paper_2602_15563_b200 import kmq
from tests import gpu_util as gu
from tests.test_gpu_launched_forms import template
from tests.test_gpu_tcgen05 import random_layer, run

pytestmark = pytest.mark.gpu
TUNED = kmq.KMQ_LAYOUT_TUNED


def check(bits, N, K, M):
    rng = np.random.default_rng(bits + N + K + M)
    idx, cb, x = random_layer(rng, N, K, bits, M)
    y_ref, s = orc.linear_f64(orc.pack_canonical(idx, bits), cb, x, K, bits)
    y = gu.gpu_linear(gu.gpu_pack(idx, bits, TUNED), cb, x, N, K, bits, TUNED)
    assert kmq.kmq_device_error_flags() == 0
    assert orc.check_linear(y, y_ref, s) <= 1.0


@pytest.mark.parametrize("bits,N,K,M,kernel", [
    (4, 700, 1528, 9, "multi"), (4, 700, 1536, 9, "tcgen05"), (4, 4095, 1032, 16, "multi"), (4, 4096, 1032, 16, "tcgen05"),
    (4, 9471, 264, 12, "multi"), (4, 9472, 264, 12, "tcgen05"), (4, 3000, 2056, 8, "tiled"),
    (2, 500, 2032, 16, "multi"), (2, 500, 2048, 16, "tcgen05"), (2, 4095, 304, 9, "multi"), (2, 4096, 304, 9, "tcgen05"),
    (1, 500, 512, 9, "tcgen05"), (1, 500, 544, 9, "multi"), (1, 9472, 8192, 16, "tcgen05"), (1, 9473, 8192, 16, "multi"),
    (1, 14080, 8160, 16, "tcgen05"), (1, 300, 800, 17, "tcgen05"), (2, 300, 1520, 17, "multi"), (2, 300, 1536, 32, "tcgen05"),
    (4, 300, 136, 32, "multi"), (4, 300, 136, 33, "tcgen05"),
])
def test_kernel_on_either_side_of_a_line(bits, N, K, M, kernel):
    assert kmq.kmq_linear_variant(N, K, bits, M, TUNED).startswith(kernel)
    check(bits, N, K, M)


@pytest.mark.parametrize("bits,N,K,M", [(4, 10230, 8192, 16), (4, 8200, 28672, 9), (2, 10240, 8192, 32), (4, 2050, 28680, 12),
                                        (2, 5130, 16400, 40), (2, 256, 512, 129), (2, 16, 64, 300), (2, 129, 640, 161),
                                        (2, 1000, 1024, 520)])
def test_shapes_that_had_another_kernel(bits, N, K, M):
    """Once balanced shapes of the multi-tile kernel and shapes of the CTA pairs."""
    (name, *_), = gu.linear_kernels(N, K, bits, M, TUNED)
    assert template(name, "linear_umma_kernel")[0] == bits
    check(bits, N, K, M)


# stages of 128 weights around the rings of 4 to 6 and the 4 groups of decoders; K that is no whole number of stages
@pytest.mark.parametrize("bits", (1, 2, 4))
@pytest.mark.parametrize("K", (128, 384, 640, 768, 800, 896, 1024, 1152, 1312, 2016))
@pytest.mark.parametrize("M", (40, 64, 90, 128))
def test_stages_around_the_ring(bits, K, M):
    check(bits, 130, K, M)


@pytest.mark.parametrize("bits", (1, 2, 4))
@pytest.mark.parametrize("N,K,M,ctas", [(130, 3328, 16, 6), (2000, 4096, 9, 4), (2500, 2048, 33, 3), (900, 2304, 96, 6),
                                        (250, 1280, 128, 3), (5000, 8192, 64, 3), (1000, 16384, 17, 6), (520, 24576, 12, 8)])
def test_clusters(bits, N, K, M, ctas):
    (name, grid, _, cluster), = gu.linear_kernels(N, K, bits, M, TUNED)
    assert template(name, "linear_umma_kernel")[0] == bits and abs(cluster - ctas) <= 2 and grid[1] == cluster
    check(bits, N, K, M)


@pytest.mark.parametrize("bits", (1, 2, 4))
def test_words_aligned_to_16_bytes_only(bits):
    """The loads of 32 bytes need more than the 16 the interface asks for."""
    N, K, M = 300, 2080, 20
    idx, cb, x = random_layer(np.random.default_rng(bits), N, K, bits, M)
    packed = gu.gpu_pack(idx, bits, TUNED)
    buf = torch.empty(packed.numel() + 16, dtype=packed.dtype, device="cuda")
    words = 16 // packed.element_size()
    off = next(o for o in range(0, 4 * words, words) if (buf.data_ptr() + o * packed.element_size()) % 32 == 16)
    odd = buf[off:off + packed.numel()]
    odd.copy_(packed)
    xd, cbd = gu.to_dev_u16(x), gu.to_dev_u16(cb)
    ys = [torch.zeros((M, N), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    for p, y in zip((packed, odd), ys):
        kmq.kmq_linear(p, cbd, xd, y, N, K, bits, M, None, 0, layout=TUNED)
    assert torch.equal(ys[0], ys[1]) and bool(ys[0].float().abs().sum() > 0)


@pytest.mark.parametrize("bits", (1, 2, 4))
@pytest.mark.parametrize("N,K,M", [(130, 128, 20000), (300, 384, 9000), (5000, 256, 1100)])
def test_pairs_on_ragged_tiles(bits, N, K, M):
    rng = np.random.default_rng(bits + N)
    idx, cb, x = random_layer(rng, N, K, bits, M)
    assert template(gu.linear_kernels(N, K, bits, M, TUNED)[0][0], "linear_umma_pair_kernel") == (bits,)
    y_ref, s = orc.linear_f64(orc.pack_canonical(idx, bits), cb, x, K, bits)
    assert orc.check_linear(run(idx, cb, x, bits), y_ref, s) <= 1.0
