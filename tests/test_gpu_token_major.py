"""GPU parity of the GEMM's token-major tile shapes (csrc/gemm_kernel.cuh; Sec. 4.2, Eq. 7).

Above 128 tokens the CTA-pair kernel with the weights in TMEM takes most launches; the token-major kernel keeps few k-blocks,
wide layers of packed codes, and 8-bit codes below K = 768.  Each shape here is checked to run it (the launch plan, also on
the CPU): single CTAs with 128- and 256-wide tiles, CTA pairs with both, gated tiles, one and several tiles a CTA, ragged
token and weight tiles, a pair whose second CTA has no tokens (596) or some (400, 203).  Accumulators must be the oracle's
integers, outputs the bits of slices of a few tokens, which run the weight-major kernel or, gated, the GEMV."""

import numpy as np
import pytest
import torch

from oracle import qvla_oracle as O
from paper_2605_28803_gb300 import qvla as Q
from tests import gpu_helpers as G

# activations (0 packed 4-bit codes, 1 the linear's operand bytes, 2 8-bit codes), M, weight rows (of each projection when
# gated), K, gated, tile shape
TILES = [
    (0, 19573, 16, 128, False, "single 128x128"), (0, 405, 4800, 1152, False, "single 128x128"),
    (0, 161, 20512, 128, False, "single 128x256"), (0, 2048, 4096, 256, False, "single 128x256"),
    (0, 29313, 16, 1024, False, "pair 256x128"), (0, 203, 29504, 1152, False, "pair 256x256"),
    (0, 400, 8192, 2048, False, "pair 256x256"), (0, 596, 5568, 2816, False, "pair 256x256"),
    (0, 455, 6528, 128, True, "single 128x256"), (0, 635, 2816, 1408, True, "single 128x256"),
    (0, 194, 14720, 1024, True, "pair 256x256"), (0, 652, 2688, 3200, True, "pair 256x256"),
    (1, 19479, 16, 128, False, "single 128x128"), (1, 322, 12928, 640, False, "single 128x128"),
    (1, 130, 19920, 128, False, "single 128x256"), (1, 1500, 4112, 128, False, "single 128x256"),
    (1, 129, 9984, 128, True, "single 128x256"), (1, 263, 13568, 128, True, "single 128x256"),
    (2, 4962, 16, 640, False, "single 128x128"), (2, 300, 3200, 512, False, "single 128x128"),
    (2, 132, 30576, 128, False, "single 128x256"), (2, 569, 12512, 256, False, "single 128x256"),
    (2, 132, 9984, 128, True, "single 128x256"), (2, 266, 4864, 384, True, "single 128x256"),
]


@pytest.mark.parametrize("codes,M,N,K,gated,shape", TILES)
def test_the_launch_plan_takes_the_token_major_kernel(codes, M, N, K, gated, shape):
    assert Q.qvla_debug_gemm_plan_codes(codes, M, K, 2 * N if gated else N, gated, 152) == (shape, 1)


@pytest.mark.gpu
@pytest.mark.parametrize("codes,M,N,K,gated,shape", TILES)
def test_tiles_are_exact(codes, M, N, K, gated, shape):
    rng = np.random.default_rng(M + N + K)
    rows = 2 * N if gated else N
    w = rng.integers(-8, 8, (rows, K)).astype(np.int8)
    wq, ws = O.pack_int4(w), (rng.uniform(0.5, 1.5, rows) / 64).astype(np.float32)
    bias = rng.standard_normal(rows).astype(np.float32)
    if gated:
        layer = Q.qvla_layer_create_gated(N, K, 128, Q.F16, Q.BF16, wq[:N], ws[:N], wq[N:], ws[N:], bias[:N], bias[N:])
    else:
        layer = Q.qvla_layer_create(N, K, 128, Q.F16, Q.BF16, wq, ws, bias)
    xs = torch.from_numpy((rng.uniform(0.5, 1.5, M) / 64).astype(np.float32)).to(G.DEV)
    nb = max(Q.qvla_linear_workspace_bytes(layer, M), Q.qvla_w4a8_workspace_bytes(layer, M))
    work = torch.empty(nb, dtype=torch.uint8, device=G.DEV)
    if codes == 1:
        x = torch.from_numpy(rng.standard_normal((M, K), dtype=np.float32)).half().to(G.DEV)
    else:
        q = rng.integers(-7, 8, (M, K)).astype(np.int8) if codes == 0 else rng.integers(-127, 128, (M, K)).astype(np.int8)
        x = torch.from_numpy(O.pack_int4(q) if codes == 0 else q).to(G.DEV)
        xsum = torch.from_numpy(q.sum(1, dtype=np.int32)).to(G.DEV)

    def run(i, m, y, acc):
        if codes == 0:
            Q.qvla_gemm_w4a4(layer, x[i:], xs[i : i + m].clone(), xsum[i : i + m].clone(), m, y, acc, G.stream())
        elif codes == 1:
            Q.qvla_w4a4_linear(layer, x[i:], m, -1, y, work, nb, G.stream())
        else:
            Q.qvla_gemm_w4a8(layer, x[i:], xs[i : i + m].clone(), m, y, acc, work, nb, G.stream())

    y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device=G.DEV)
    acc = None if codes == 1 else torch.full((M, rows), -(2 ** 31), dtype=torch.int32, device=G.DEV)
    run(0, M, y, acc)
    Q.qvla_check_device(G.stream())
    if codes != 1:
        ref = O.int_gemm(q, w)
        assert np.array_equal(acc.cpu().numpy(), ref)
    if codes == 2 and gated:  # no other kernel of few tokens takes these: the oracle's epilogue
        gate, up = (O.dequant_output(ref[:, s], xs.cpu().numpy(), ws[s], bias[s], "bf16") for s in (slice(0, N), slice(N, rows)))
        G.assert_output_close(y.double().cpu().numpy(), O.round_to_format(O.gated_glue(gate, up), "bf16"), "bf16")
    else:
        want = torch.empty_like(y)
        step = 4 if gated else 128
        for i in range(0, M, step):
            run(i, min(step, M - i), want[i:], None)
        Q.qvla_check_device(G.stream())
        assert torch.equal(y, want)
    layer.close()
