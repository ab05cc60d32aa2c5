"""The multi-tile kernel at b = 4, up to 16 batch rows (half of a tile's rows from pair tables): every shape of CTA, ragged
tiles and row lengths."""
import numpy as np
import pytest

from oracle import kmq_oracle as orc
from paper_2602_15563_b200 import kmq
from tests import gpu_util as gu
from tests.test_gpu_tcgen05 import random_layer

pytestmark = pytest.mark.gpu
TUNED = kmq.KMQ_LAYOUT_TUNED


@pytest.mark.parametrize("N,K,M", [(17, 136, 9), (100, 4160, 16), (3000, 4096, 11), (5000, 392, 16), (8190, 264, 4),
                                   (9000, 1032, 8), (10001, 776, 15), (20000, 520, 16)])
def test_half_tables(N, K, M):
    rng = np.random.default_rng(N + K + M)
    idx, cb, x = random_layer(rng, N, K, 4, M)
    y_ref, s = orc.linear_f64(orc.pack_canonical(idx, 4), cb, x, K, 4)
    y = gu.gpu_linear(gu.gpu_pack(idx, 4, TUNED), cb, x, N, K, 4, TUNED)
    ratio = orc.check_linear(y, y_ref, s)
    assert ratio <= 1.0, f"error/tolerance = {ratio} [{kmq.kmq_linear_variant(N, K, 4, M, TUNED)}]"
