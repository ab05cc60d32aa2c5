"""kmq_linear_host with pinned and pageable, aligned and unaligned buffers, below and above the size that a kernel copies."""
import pytest
import torch

from paper_2602_15563_b200 import kmq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pinned", (True, False))
@pytest.mark.parametrize("offset", (0, 1))
@pytest.mark.parametrize("N,K,M", [(1, 32, 1), (13, 64, 1), (1000, 2880, 3), (4096, 4096, 32), (4096, 4096, 33)])
def test_host_buffers(N, K, M, offset, pinned):
    bits, layout = 1, kmq.KMQ_LAYOUT_TUNED
    g = torch.Generator().manual_seed(N + M)
    packed = torch.randint(-2**31, 2**31 - 1, (kmq.kmq_packed_bytes(N, K, bits, layout) // 4,), dtype=torch.int32,
                           generator=g).cuda()
    cb = torch.randn((N, 2), generator=g).to(torch.bfloat16).cuda()
    xh = torch.empty(M * K + 16, dtype=torch.bfloat16, pin_memory=pinned)
    yh = torch.zeros(M * N + 16, dtype=torch.bfloat16, pin_memory=pinned)
    xh.copy_(torch.randn(M * K + 16, generator=g).to(torch.bfloat16))
    x = torch.zeros((M, K), dtype=torch.bfloat16, device="cuda")
    y, y2 = (torch.zeros((M, N), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    nbytes = kmq.kmq_workspace_bytes(N, K, bits, M, layout)
    ws = torch.empty(max(nbytes, 16), dtype=torch.uint8, device="cuda")
    kmq.kmq_linear_host(packed, cb, xh.data_ptr() + 2 * offset, yh.data_ptr() + 2 * offset, N, K, bits, M, x, y, ws, nbytes,
                        layout=layout)
    assert torch.equal(x.cpu().flatten().view(torch.int16), xh[offset:offset + M * K].view(torch.int16))
    kmq.kmq_linear(packed, cb, x, y2, N, K, bits, M, ws, nbytes, layout=layout)
    got = yh[offset:offset + M * N].view(torch.int16)
    assert torch.equal(got, y2.cpu().flatten().view(torch.int16))
    assert not yh[:offset].any() and not yh[offset + M * N:].any()
