"""The fit by buckets where it can go wrong: row lengths around the padded sizes, row lengths that are no multiple of
four, values outside the octaves the buckets resolve, rows on either side of the limits that send a row to the sorting
path, and the packing fused behind the fit with padding in every layout."""
import numpy as np
import pytest
import torch

from oracle import kmq_quant_oracle as qorc
from paper_2602_15563_b200 import kmq
from tests import gpu_util as gu
from tests.test_gpu_quantize import check_fit

pytestmark = pytest.mark.gpu
C, T, L = kmq.KMQ_LAYOUT_CANONICAL, kmq.KMQ_LAYOUT_TUNED, kmq.KMQ_LAYOUT_TABLE


@pytest.mark.parametrize("bits", (1, 4))
@pytest.mark.parametrize("K", (31, 127, 1023, 2048, 2049, 8190, 8193, 16385, 32767))
def test_row_lengths(K, bits):
    rng = np.random.default_rng(K + bits)
    check_fit((rng.standard_normal((3, K)) * 0.02).astype(np.float32), bits)


@pytest.mark.parametrize("bits", (1, 2, 4))
def test_values_of_all_magnitudes(bits):
    """Mixed buckets filled (tiny values, far outliers, subnormals, zeros), up to and over their limit."""
    rng = np.random.default_rng(bits)
    K = 2048
    base = rng.standard_normal((8, K)) * 0.02
    base[0, :200] *= 2.0 ** -rng.integers(10, 100, 200)            # below the range, both signs
    base[1, :60] *= 2.0 ** rng.integers(6, 14, 60)                 # above it
    base[2, :300] *= 2.0 ** -20                                    # within the limit per sign
    base[3, :1200] *= 2.0 ** -20                                   # over it: sorted
    base[4] *= 2.0 ** -130                                         # subnormal rows
    base[5, ::2] = 0.0
    base[6] = np.abs(base[6]) + 1.0                                # one sign, two octaves, crowded
    base[7] = np.round(base[7] * 400) / 400                        # few distinct values
    check_fit(base.astype(np.float32), bits)


@pytest.mark.parametrize("n_same", (380, 390))
def test_bucket_limit(n_same):
    rng = np.random.default_rng(n_same)
    W = rng.standard_normal((2, 4096)).astype(np.float32)
    W[0, :n_same] = np.float32(1.3) + np.arange(n_same, dtype=np.float32) * np.float32(2.0 ** -20)
    check_fit(W, 4)


@pytest.mark.parametrize("bits", (1, 2, 4))
@pytest.mark.parametrize("layout", (C, T, L))
@pytest.mark.parametrize("N,K", ((1, 32), (17, 288), (33, 1056), (5, 8224)))
def test_fused_packing(N, K, layout, bits):
    rng = np.random.default_rng(N + K + bits)
    W = (rng.standard_normal((N, K)) * 0.02).astype(np.float32)
    if N > 16:
        W[16] = np.where(np.arange(K) % 2 == 0, 0.25, -0.5)        # fewer distinct values than centroids
    d_w = torch.from_numpy(W).cuda()
    cb = torch.empty(N * (1 << bits) + 8, dtype=torch.int16, device="cuda")
    nbytes = kmq.kmq_packed_bytes(N, K, bits, layout)
    buf, off = gu.dev_bytes(nbytes)
    kmq.kmq_quantize_rows(d_w, N, K, bits, 20, layout, cb, buf.data_ptr() + off)
    torch.cuda.synchronize()
    assert gu.canaries_intact(buf, off, nbytes)
    got_cb = cb[:N * (1 << bits)].cpu().numpy().view(np.uint16).reshape(N, -1)
    np.testing.assert_array_equal(got_cb, qorc.centroids_to_bf16(qorc.lloyd_rows(W, bits)))
    want = gu.gpu_pack(qorc.nearest_centroid(W, got_cb), bits, layout)
    assert torch.equal(buf[off:off + nbytes].view(torch.int32), want)
