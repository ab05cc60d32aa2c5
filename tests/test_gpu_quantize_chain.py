"""Quantiser and layer in turn on one stream, without synchronisation, into the same buffers of indices, codebooks and
scales: the layer's kernels read these before they wait for the previous kernel (programmatic dependent launch), which is
sound only because the kernels that write them never release their dependents early.  A layer that read too early would see
the weights of the round before."""
import pytest
import torch

from paper_2602_15563_b200 import kmq

pytestmark = pytest.mark.gpu
C, T, L = kmq.KMQ_LAYOUT_CANONICAL, kmq.KMQ_LAYOUT_TUNED, kmq.KMQ_LAYOUT_TABLE
N, K, ROUNDS = 1040, 4096, 6


def in_turn(step, sync):
    """step(i) enqueues round i and returns its output; all rounds on one stream."""
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    outs = []
    with torch.cuda.stream(stream):
        for i in range(ROUNDS):
            outs.append(step(i))
            if sync:
                stream.synchronize()
    stream.synchronize()
    return outs


def weights(seed, M=2):
    g = torch.Generator(device="cuda").manual_seed(seed)
    W = [torch.randn(N, K, device="cuda", generator=g) * (0.02 * (i + 1)) for i in range(ROUNDS)]
    return W, torch.randn(M, K, device="cuda", generator=g).to(torch.bfloat16)


def check(step):
    ref = in_turn(step, True)
    assert all(not torch.equal(a, b) for a, b in zip(ref, ref[1:]))
    for _ in range(3):
        for a, b in zip(in_turn(step, False), ref):
            assert torch.equal(a, b)
    assert kmq.kmq_device_error_flags() == 0


@pytest.mark.parametrize("bits,layout", [(1, T), (2, T), (4, T), (1, L), (2, L), (2, C), (4, C)])
def test_quantize_rows_then_linear(bits, layout):
    W, x = weights(bits)
    M = x.shape[0]
    packed = torch.zeros(kmq.kmq_packed_bytes(N, K, bits, layout) // 4, dtype=torch.int32, device="cuda")
    cb = torch.zeros(N, 1 << bits, dtype=torch.bfloat16, device="cuda")
    nbytes = kmq.kmq_workspace_bytes(N, K, bits, M, layout)
    ws = torch.empty(max(nbytes, 16), dtype=torch.uint8, device="cuda")
    y = torch.zeros(ROUNDS, M, N, dtype=torch.bfloat16, device="cuda")

    def step(i):
        kmq.kmq_quantize_rows(W[i], N, K, bits, 5, layout, cb, packed)
        kmq.kmq_linear(packed, cb, x, y[i], N, K, bits, M, ws, nbytes, layout=layout)
        return y[i].clone()

    check(step)


@pytest.mark.parametrize("bits", (1, 2, 4))
@pytest.mark.parametrize("M", (12, 40, 100, 200))
@pytest.mark.parametrize("forced", (False, True))
def test_quantize_rows_then_tcgen05(bits, M, forced):
    """The kernel that reads packed words and codebooks of 128 rows ahead of its wait, by kmq_linear's choice and by its own
    entry point."""
    W, x = weights(20 + bits, M)
    assert kmq.kmq_linear_variant(N, K, bits, M, T).startswith("tcgen05") and kmq.kmq_workspace_bytes(N, K, bits, M, T) == 0
    packed = torch.zeros(kmq.kmq_packed_bytes(N, K, bits, T) // 4, dtype=torch.int32, device="cuda")
    cb = torch.zeros(N, 1 << bits, dtype=torch.bfloat16, device="cuda")
    y = torch.zeros(ROUNDS, M, N, dtype=torch.bfloat16, device="cuda")

    def step(i):
        kmq.kmq_quantize_rows(W[i], N, K, bits, 5, T, cb, packed)
        if forced:
            kmq.kmq_linear_tcgen05(packed, cb, x, y[i], N, K, bits, M)
        else:
            kmq.kmq_linear(packed, cb, x, y[i], N, K, bits, M, None, 0, layout=T)
        return y[i].clone()

    check(step)


@pytest.mark.parametrize("bits", (1, 2, 4))
@pytest.mark.parametrize("table", (False, True))
def test_quantize_block_then_linear(bits, table):
    W, x = weights(10 + bits)
    M = x.shape[0]
    scales = torch.zeros(N, K // 64, dtype=torch.bfloat16, device="cuda")
    cb = torch.zeros(1 << bits, dtype=torch.bfloat16, device="cuda")
    wq = torch.zeros(kmq.kmq_block_packed_bytes(N, K, bits), dtype=torch.uint8, device="cuda")
    sample = torch.zeros(8192, dtype=torch.float32, device="cuda")
    tab = torch.zeros(kmq.kmq_block_table_bytes(N, K, bits), dtype=torch.uint8, device="cuda")
    nbytes = kmq.kmq_block_table_workspace_bytes(N, K, bits)
    ws = torch.empty(max(nbytes, 16), dtype=torch.uint8, device="cuda")
    y = torch.zeros(ROUNDS, M, N, dtype=torch.bfloat16, device="cuda")

    def step(i):
        kmq.kmq_block_quantize(W[i], N, K, bits, kmq.KMQ_LAMBDA_ABSMAX, 5, 8192, scales, cb, wq, sample)
        if table:
            kmq.kmq_block_table_pack(wq, scales, N, K, bits, tab)
            kmq.kmq_block_table_linear(tab, cb, x, y[i], N, K, bits, M, ws, nbytes)
        else:
            kmq.kmq_block_linear(wq, scales, cb, x, y[i], N, K, bits, M)
        return y[i].clone()

    check(step)


@pytest.mark.parametrize("mode", (kmq.KMQ_LAMBDA_ABSMAX, kmq.KMQ_LAMBDA_ABSMEAN))
def test_quantize_block_in_a_graph(mode):
    """The kernels of a call start beside one another: captured, calls in turn on the same sample and scales give what they give
    one at a time."""
    W, _ = weights(40)
    bits = 4
    scales = torch.zeros(N, K // 64, dtype=torch.bfloat16, device="cuda")
    sample = torch.zeros(8192, dtype=torch.float32, device="cuda")
    cb = torch.zeros(ROUNDS, 1 << bits, dtype=torch.bfloat16, device="cuda")
    wq = torch.zeros(ROUNDS, kmq.kmq_block_packed_bytes(N, K, bits), dtype=torch.uint8, device="cuda")

    def all_rounds(sync):
        for i in range(ROUNDS):
            kmq.kmq_block_quantize(W[i], N, K, bits, mode, 5, 8192, scales, cb[i], wq[i], sample)
            if sync:
                torch.cuda.synchronize()

    all_rounds(True)
    want = cb.clone(), wq.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        all_rounds(False)
    for _ in range(2):
        cb.zero_()
        wq.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(cb, want[0]) and torch.equal(wq, want[1])
