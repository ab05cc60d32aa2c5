"""The nearest of 16 centroids through a grid of cells: weights on and one step beside the midpoints, codebooks whose
midpoints share cells, coincide or span many magnitudes, against the exact comparison of oracle/kmq_quant_oracle.py (indices
equal, no tolerance); arrays that are aligned to 16 bytes and not to 32, whose loads are narrower, against aligned ones."""
import numpy as np
import pytest
import torch

from oracle import kmq_block_oracle as blk
from oracle import kmq_quant_oracle as qorc
from paper_2602_15563_b200 import kmq
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def codebook(kind):
    i = np.arange(16)
    c = {"even": -1 + i / 7.5, "normal": np.sinh((i - 7.5) / 4), "one far": np.append(i[:15] * 1e-3, 1.0),
         "equal": np.repeat([-1.0, -0.25, 0.5, 1.0], 4), "constant": np.full(16, 0.25), "octaves": 2.0 ** (i - 15),
         "dyadic": (i - 8) / 8.0, "tiny": (i - 8) * 2.0 ** -100}[kind]
    return qorc.f32_to_bf16_rne(c.astype(np.float32))


def around(values, rng, count):
    """float32 values at, one step below and one above the given ones, and random ones between."""
    v = np.concatenate([np.nextafter(values, -np.inf), values, np.nextafter(values, np.inf)]).astype(np.float32)
    span = float(np.abs(values).max()) * 1.5 + 1e-30
    fill = rng.uniform(-span, span, count - v.size).astype(np.float32)
    return rng.permutation(np.concatenate([v, fill]))


@pytest.mark.parametrize("kind", ("even", "normal", "one far", "equal", "constant", "octaves", "dyadic", "tiny"))
def test_block_assignment_on_the_midpoints(kind):
    N, K, rng = 6, 512, np.random.default_rng(3)
    cb = codebook(kind)
    c = blk._bf16_to_f64(cb)
    mids = (0.5 * (c[1:] + c[:-1])).astype(np.float32)
    scale_bits = qorc.f32_to_bf16_rne(np.float32([1.0, 0.5, 0.3, 7.25, 2e-31, 3e30]))   # the last two beyond the grid's range
    scales = np.repeat(scale_bits[:, None], K // 64, axis=1)
    s = blk._bf16_to_f64(scale_bits)
    with np.errstate(over="ignore"):
        W = np.stack([around((mids * np.float64(s[n])).astype(np.float32), rng, K) for n in range(N)])
    W = np.nan_to_num(W, posinf=1e38, neginf=-1e38).astype(np.float32)
    out = torch.empty(kmq.kmq_block_packed_bytes(N, K, 4), dtype=torch.uint8, device="cuda")
    kmq.kmq_block_assign_pack(torch.from_numpy(W).cuda(), gu.to_dev_u16(scales), gu.to_dev_u16(cb), N, K, 4, out)
    got = blk.unpack_bytes(out.cpu().numpy().reshape(N, -1), K, 4)
    assert np.array_equal(got, qorc.block_assign(W, scales, cb))


@pytest.mark.parametrize("K", (32, 512, 992, 1024, 4096))
def test_rows_whose_thresholds_share_cells(K):
    rng = np.random.default_rng(K)
    W = rng.standard_normal((5, K)).astype(np.float32)
    W[1] = rng.choice(np.float32([-1, -0.5, 0.125, 3]), K)                 # fewer values than centroids
    W[2] *= np.exp2(rng.integers(-12, 12, K)).astype(np.float32)           # most thresholds in one cell
    W[3, 0] = 1e4
    W[4] = np.round(W[4] * 8) / 8                                          # weights on the midpoints
    cb = torch.empty((5, 16), dtype=torch.bfloat16, device="cuda")
    packed = torch.empty(kmq.kmq_packed_bytes(5, K, 4, kmq.KMQ_LAYOUT_TUNED) // 4, dtype=torch.int32, device="cuda")
    kmq.kmq_quantize_rows(torch.from_numpy(W).cuda(), 5, K, 4, 20, kmq.KMQ_LAYOUT_TUNED, cb, packed)
    got = gu.gpu_unpack(packed, 5, K, 4, kmq.KMQ_LAYOUT_TUNED)
    assert np.array_equal(got, qorc.nearest_centroid(W, cb.view(torch.int16).cpu().numpy().view(np.uint16)))


@pytest.mark.parametrize("bits", (1, 2, 4))
def test_weights_aligned_to_16_bytes_only(bits):
    N, K = 17, 1088
    buf = torch.randn(N * K + 8, device="cuda", generator=torch.Generator(device="cuda").manual_seed(bits))
    results = []
    for off in (4, 0):
        W = buf[off:off + N * K]
        if off == 0:
            W.copy_(buf[4:4 + N * K].clone())
        cb = torch.empty((N, 1 << bits), dtype=torch.bfloat16, device="cuda")
        packed = torch.empty(kmq.kmq_packed_bytes(N, K, bits, kmq.KMQ_LAYOUT_TUNED) // 4, dtype=torch.int32, device="cuda")
        kmq.kmq_quantize_rows(W, N, K, bits, 20, kmq.KMQ_LAYOUT_TUNED, cb, packed)
        scales = torch.empty((N, K // 64), dtype=torch.bfloat16, device="cuda")
        shared = torch.empty(1 << bits, dtype=torch.bfloat16, device="cuda")
        wq = torch.empty(kmq.kmq_block_packed_bytes(N, K, bits), dtype=torch.uint8, device="cuda")
        sample = torch.empty(4096, dtype=torch.float32, device="cuda")
        kmq.kmq_block_quantize(W, N, K, bits, kmq.KMQ_LAMBDA_ABSMAX, 20, 4096, scales, shared, wq, sample)
        results.append([t.clone() for t in (cb, packed, scales, shared, wq)])
    assert all(torch.equal(a, b) for a, b in zip(*results))


@pytest.mark.parametrize("K", (248, 256, 264))
@pytest.mark.parametrize("layout", (kmq.KMQ_LAYOUT_CANONICAL, kmq.KMQ_LAYOUT_TUNED))
def test_rows_at_the_length_from_which_cells_are_used(K, layout):
    W = (np.random.default_rng(K).standard_normal((37, K)) * 0.02).astype(np.float32)
    cb = torch.empty((37, 16), dtype=torch.bfloat16, device="cuda")
    packed = torch.empty(kmq.kmq_packed_bytes(37, K, 4, layout) // 4, dtype=torch.int32, device="cuda")
    kmq.kmq_quantize_rows(torch.from_numpy(W).cuda(), 37, K, 4, 20, layout, cb, packed)
    got = gu.gpu_unpack(packed, 37, K, 4, layout)
    assert np.array_equal(got, qorc.nearest_centroid(W, cb.view(torch.int16).cpu().numpy().view(np.uint16)))
