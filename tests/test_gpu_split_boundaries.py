"""The balanced split where every cut falls on a tile boundary (tiles a multiple of the CTAs): its second kernel has
nothing to add, and the next layer must all the same see the finished output of the first."""
import numpy as np
import pytest
import torch

from oracle import kmq_oracle as orc
from paper_2602_15563_b200 import kmq
from tests.test_gpu_chain import build_chain, run_chain

pytestmark = pytest.mark.gpu
T = kmq.KMQ_LAYOUT_TUNED
SLOT_BYTES = 2 * (16 * 8 + 8) * 4      # scratch of one CTA


def test_next_layer_sees_finished_output():
    K, bits, M = 16384, 4, 1
    ctas = kmq.kmq_workspace_bytes(1 << 16, K, bits, M, T) // SLOT_BYTES
    N = 2 * ctas * 16
    assert kmq.kmq_linear_variant(N, K, bits, M, T).startswith("split")
    assert kmq.kmq_workspace_bytes(N, K, bits, M, T) == ctas * SLOT_BYTES and ctas > 0
    layers = build_chain([K, N, 2048], [(bits, T), (2, T)], M, seed=3)
    g = torch.Generator(device="cuda").manual_seed(4)
    x0 = torch.randn(M * K, device="cuda", generator=g).to(torch.bfloat16).view(torch.int16)
    ref = run_chain(layers, x0, M, sync=True)
    for _ in range(5):
        for a, b in zip(run_chain(layers, x0, M, sync=False), ref):
            assert torch.equal(a, b)
    rows = np.arange(0, N, 397)
    packed = orc.pack_canonical(layers[0]["idx"][torch.from_numpy(rows).cuda()].cpu().numpy(), bits)
    y_ref, s = orc.linear_f64(packed, layers[0]["cb"].cpu().numpy().view(np.uint16)[rows],
                              x0.cpu().numpy().view(np.uint16).reshape(M, K), K, bits)
    assert orc.check_linear(ref[0].cpu().numpy().view(np.uint16).reshape(M, N)[:, rows], y_ref, s) <= 1.0
