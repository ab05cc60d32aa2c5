"""kmq_dequant_to_bf16 where a warp's share of a row (128 chunks of 8 weights) begins and ends: rows of one chunk, of one share and
a chunk less or more, of several; fewer shares than a CTA has warps; every layout, bit for bit."""
import numpy as np
import pytest
import torch

from oracle import kmq_oracle as orc
from paper_2602_15563_b200 import kmq
from tests import gpu_util as gu
from tests.test_gpu_tcgen05 import random_layer

pytestmark = pytest.mark.gpu
LAYOUTS = (kmq.KMQ_LAYOUT_CANONICAL, kmq.KMQ_LAYOUT_TUNED, kmq.KMQ_LAYOUT_TABLE)


@pytest.mark.parametrize("layout", LAYOUTS)
@pytest.mark.parametrize("bits", (1, 2, 4))
@pytest.mark.parametrize("N,K", [(1, 32), (7, 992), (9, 1024), (3, 1056), (33, 2048), (2, 3104), (17, 288)])
def test_shares_of_a_row(N, K, bits, layout):
    rng = np.random.default_rng(N + K + bits)
    idx, cb, _ = random_layer(rng, N, K, bits, 1)
    packed = gu.gpu_pack(idx, bits, layout)
    buf, off = gu.dev_bytes(N * K * 2)
    kmq.kmq_dequant_to_bf16(packed, gu.to_dev_u16(cb), buf.data_ptr() + off, N, K, bits, layout=layout)
    torch.cuda.synchronize()
    assert gu.canaries_intact(buf, off, N * K * 2)
    got = buf[off:off + N * K * 2].cpu().numpy().view(np.uint16).reshape(N, K)
    assert np.array_equal(got, orc.dequant_bits(orc.pack_canonical(idx, bits), cb, K, bits))
