"""Prefill batches (M > 128).  The CTA-pair kernel at its edges, on shapes of which the test sees that they reach it: one row block
of the pair empty or ragged, batch tiles of 160 to 256 rows that do not divide M, K shorter than the ring, shorter than a stage
and no whole number of stages or steps.  Smaller shapes, most of which are batch tiles of the single-CTA kernel."""
import numpy as np
import pytest

from oracle import kmq_oracle as orc
from paper_2602_15563_b200 import kmq
from tests import gpu_util as gu
from tests.test_gpu_launched_forms import template
from tests.test_gpu_tcgen05 import random_layer, run

pytestmark = pytest.mark.gpu
T = kmq.KMQ_LAYOUT_TUNED


@pytest.mark.parametrize("bits", (1, 2, 4))
@pytest.mark.parametrize("N,Kmul,M", [(256, 4, 129), (16, 1, 300), (128, 9, 160), (129, 5, 161), (257, 33, 256),
                                      (520, 17, 257), (1000, 8, 520), (2048, 3, 700), (5000, 2, 1100)])
def test_small_prefill_matches_oracle(bits, N, Kmul, M):
    K = (128 // bits) * Kmul
    rng = np.random.default_rng(100 * bits + N + M)
    idx, cb, x = random_layer(rng, N, K, bits, M)
    y_ref, s = orc.linear_f64(orc.pack_canonical(idx, bits), cb, x, K, bits)
    ratio = orc.check_linear(run(idx, cb, x, bits), y_ref, s)
    assert ratio <= 1.0, f"error/tolerance = {ratio}"
    assert kmq.kmq_linear_variant(N, K, bits, M, T).startswith("tcgen05")
    assert kmq.kmq_linear_num_launches(N, K, bits, M, T) == 1
    y2 = gu.gpu_linear(gu.gpu_pack(idx, bits, T), cb, x, N, K, bits, T)
    assert orc.check_linear(y2, y_ref, s) <= 1.0
    assert kmq.kmq_device_error_flags() == 0


# `units`: packed words by which a row is longer than `K` weights.  Rows per batch tile: 160, 192, 160, 160, 192, 256, 160, 256.
@pytest.mark.parametrize("bits", (1, 2, 4))
@pytest.mark.parametrize("N,K,units,M", [(9489, 256, 1, 129), (9600, 512, 1, 161), (9700, 1280, -1, 160), (6290, 512, 1, 257),
                                         (3800, 1024, -1, 520), (9489, 256, -1, 256), (6300, 64, 0, 300), (3100, 384, 0, 700)])
def test_pair_kernel_at_its_edges(bits, N, K, units, M):
    K += units * (32 // bits)
    (name, _, _, cluster), = gu.linear_kernels(N, K, bits, M, T)
    assert template(name, "linear_umma_pair_kernel") == (bits,) and cluster == 2
    idx, cb, x = random_layer(np.random.default_rng(N + M + bits), N, K, bits, M)
    y_ref, s = orc.linear_f64(orc.pack_canonical(idx, bits), cb, x, K, bits)
    y = gu.gpu_linear(gu.gpu_pack(idx, bits, T), cb, x, N, K, bits, T)
    assert kmq.kmq_device_error_flags() == 0
    assert orc.check_linear(y, y_ref, s) <= 1.0


@pytest.mark.parametrize("N,K,M", [(384, 2048, 300), (2100, 4096, 200), (4096, 1024, 512)])
def test_several_batch_tiles_of_the_single_cta_kernel(N, K, M):
    """Shapes with too few 256 x 256 tiles for the pairs: batch tiles of 128 rows in one launch, K split over clusters."""
    rng = np.random.default_rng(N + M)
    idx, cb, x = random_layer(rng, N, K, 2, M)
    y_ref, s = orc.linear_f64(orc.pack_canonical(idx, 2), cb, x, K, 2)
    assert orc.check_linear(run(idx, cb, x, 2), y_ref, s) <= 1.0
