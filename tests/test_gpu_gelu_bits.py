"""Gated layers: the bits of h = gelu(gate) * up at values next to a rounding boundary (Sec. 4.2's glue, tanh GELU).

A next layer's 4-bit codes follow the last bit of h, so h is pinned to the bit: the pairs below are those where the same
function with its exponential's argument folded into one polynomial (about an ulp of float32 away) rounds to the other
neighbour.  Tokens of zeros make gate and up the layer's biases exactly, in every kernel that a gated layer takes: the decode
GEMV in one launch and on packed codes, the CTA-pair kernel on operand bytes and on packed codes, and 8-bit codes."""

import numpy as np
import pytest
import torch

from paper_2605_28803_gb300 import qvla as Q
from tests import gpu_helpers as G

pytestmark = pytest.mark.gpu

# (gate, up, h) as the bits of the 16-bit types
F16 = [
    (0x2ABB, 0x3DD7, 0x291E), (0x38AF, 0x3EF3, 0x39DE), (0xA609, 0x3FFA, 0xA5E8), (0xB388, 0x3EE9, 0xB14B),
    (0xB6B2, 0x3EAB, 0xB38A), (0xB90E, 0x3CA5, 0xB231), (0xBA08, 0x3D17, 0xB2ED), (0xBB40, 0x3D08, 0xB2A8),
    (0xBC56, 0x3C1D, 0xB0F8), (0xBCE0, 0x3F36, 0xB3DA), (0xBD24, 0x3F93, 0xB3C0), (0xBD62, 0x3CE7, 0xB0B7),
    (0xBEA3, 0x3C1D, 0xAD4F), (0xBF10, 0x3D9F, 0xAE29), (0xBF4D, 0x3F3A, 0xAF2D), (0xBFE7, 0x3ED4, 0xAD32),
    (0xC033, 0x3FDF, 0xACB4), (0xC059, 0x3D88, 0xA9AC), (0xC07E, 0x3D9E, 0xA8EE), (0xC0B6, 0x3D3C, 0xA72D),
    (0xC0D6, 0x3E9D, 0xA7D0), (0xC115, 0x3F84, 0xA689), (0xC144, 0x3C44, 0xA1D4), (0xC16C, 0x3D91, 0xA225),
    (0xC1A0, 0x3CEA, 0xA00E), (0xC1F1, 0x3C3F, 0x9C57), (0xC217, 0x3F5B, 0x9DED), (0xC229, 0x3E58, 0x9C8E),
    (0xC288, 0x3C3B, 0x966E), (0xC2B9, 0x3C93, 0x94E7), (0xC2F1, 0x3D50, 0x9385), (0xC308, 0x3FBA, 0x9496),
    (0xC335, 0x3F4E, 0x9215), (0xC355, 0x3D16, 0x8E89), (0xC39A, 0x3DDF, 0x8C39), (0xC3A4, 0x3CFD, 0x8A93),
    (0xC3EE, 0x3FE3, 0x895D), (0xC40A, 0x3D37, 0x84FA), (0xC411, 0x3D7C, 0x8495), (0xC491, 0x3F98, 0x8070)]
BF16 = [
    (0x3EBD, 0x3FAD, 0x3EA4), (0xBF63, 0x3FD9, 0xBE91), (0xBF68, 0x3FB8, 0xBE73), (0xC067, 0x3FCE, 0xBA27),
    (0xC071, 0x3F84, 0xB95E), (0xC0D1, 0x3FE6, 0xAB65), (0xC0DC, 0x3FF5, 0xA8AE), (0xC0ED, 0x3FD1, 0xA3D4)]


@pytest.mark.parametrize("dt", ["f16", "bf16"])
@pytest.mark.parametrize("M", [1, 2, 5, 200])
def test_gelu_glue_is_pinned_to_the_bit(dt, M):
    t, code, rows = {"f16": (torch.float16, Q.F16, F16), "bf16": (torch.bfloat16, Q.BF16, BF16)}[dt]
    bits = torch.tensor(rows, dtype=torch.int32).to(torch.int16)
    gate, up, want = (bits[:, i].contiguous().view(t) for i in range(3))
    H, K = 128, 256  # a whole ring stage of the CTA-pair kernel
    n = len(rows)
    b = [np.zeros(H, np.float32) for _ in range(2)]
    for dst, v in zip(b, (gate, up)):
        dst[:n] = v.float().numpy()
    wq = np.random.default_rng(M).integers(0, 256, (H, K // 2), dtype=np.uint8)
    ws = np.full(H, 0.01, np.float32)
    layer = Q.qvla_layer_create_gated(H, K, 128, code, code, wq, ws, wq, ws, b[0], b[1])
    x = torch.zeros(M, K, dtype=t, device=G.DEV)
    nb = Q.qvla_linear_workspace_bytes(layer, M)
    work = torch.empty(max(nb, Q.qvla_w4a8_workspace_bytes(layer, M)), dtype=torch.uint8, device=G.DEV)
    xq = torch.zeros(M, K // 2, dtype=torch.uint8, device=G.DEV)
    xs, xsum = torch.zeros(M, device=G.DEV), torch.zeros(M, dtype=torch.int32, device=G.DEV)
    calls = [lambda y: Q.qvla_w4a4_linear(layer, x, M, -1, y, work, nb, G.stream()),
             lambda y: Q.qvla_gemm_w4a4(layer, xq, xs, xsum, M, y, None, G.stream()),
             lambda y: Q.qvla_w4a8_linear(layer, x, M, -1, y, work, work.numel(), G.stream())]
    for call in calls:
        y = torch.full((M, H), float("nan"), dtype=t, device=G.DEV)
        call(y)
        Q.qvla_check_device(G.stream())
        assert torch.equal(y.cpu().view(torch.int16)[:, :n], want.view(torch.int16).expand(M, n))
    layer.close()
