"""Error of the fp32 sums of the tcgen05 kernel: a tcgen05.mma cuts its sum off, so that an accumulator's error grows with the
number of MMAs that add into it; the slices of K take turns on 8 accumulators (up to 16 batch rows), 4 (up to 32) or 2.

Bound.  One of L MMAs that add into an accumulator loses half a unit of 2^-23 of the partial sum on average, and the partial
sums of random terms are about 0.7 of the final one: 0.35 L 2^-23 of the result, of the same sign throughout.  With A
accumulators that are shorter by A and smaller by sqrt(A), and whose errors add up as their signs do, it is 1 / A of that.  Such
an error moves a result to a neighbouring bf16 value, on average 2^-7.5 of the result away, with a probability of the error
over that distance: 0.35 2^-15.5 L / A = 7.6e-6 L / A of all results are not the rounded exact ones.  Half as much again is allowed, and
1e-4 for few MMAs, where the sum over the accumulators and the cluster counts too."""
import pytest
import torch

from paper_2602_15563_b200 import kmq

pytestmark = pytest.mark.gpu
T = kmq.KMQ_LAYOUT_TUNED


def layer(bits, N, K, M):
    g = torch.Generator(device="cuda").manual_seed(bits + N + K + M)
    idx = torch.randint(0, 1 << bits, (N, K), dtype=torch.uint8, device="cuda", generator=g)
    cb = (torch.randn(N, 1 << bits, device="cuda", generator=g) * 0.02).sort(dim=1).values.to(torch.bfloat16)
    x = torch.randn(M, K, device="cuda", generator=g).to(torch.bfloat16)
    exact = torch.cat([x.double() @ cb[i:i + 1024].double().gather(1, idx[i:i + 1024].long()).T for i in range(0, N, 1024)], 1)
    packed = torch.empty(kmq.kmq_packed_bytes(N, K, bits, T) // 4, dtype=torch.int32, device="cuda")
    kmq.kmq_pack(idx, N, K, bits, packed, layout=T)
    return packed, cb, x, exact


@pytest.mark.parametrize("bits,N,K,M", [(4, 12288, 8192, 16), (2, 8192, 28672, 9), (1, 8192, 28672, 16), (4, 8192, 28672, 32),
                                        (2, 12288, 8192, 24), (4, 12288, 8192, 48), (1, 8192, 28672, 64), (2, 12288, 8192, 90),
                                        (4, 12288, 8192, 128), (4, 4096, 2048, 128)])
def test_share_of_results_that_are_not_the_rounded_exact_ones(bits, N, K, M):
    packed, cb, x, exact = layer(bits, N, K, M)
    y = torch.zeros(M, N, dtype=torch.bfloat16, device="cuda")
    kmq.kmq_linear_tcgen05(packed, cb, x, y, N, K, bits, M)
    off = float((y != exact.float().to(torch.bfloat16)).float().mean())
    assert kmq.kmq_device_error_flags() == 0
    assert off <= 1.5 * 7.6e-6 * (K / 16) / (8 if M <= 16 else 4 if M <= 32 else 2) + 1e-4
