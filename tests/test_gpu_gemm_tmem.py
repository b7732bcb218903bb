"""GPU parity of the GEMM on CTA pairs with the expanded weights in TMEM (csrc/gemm_tmem.cu; Sec. 4.2, Eq. 7).

qvla_w4a4_linear's GEMM takes it for batches of more than 128 tokens and for gated layers from 5 (below K = 768 where it is
estimated faster); qvla_gemm_w4a4 takes packed codes there where it is estimated faster, else to the token-major kernel, and
expands them in its converters.  Every accumulation is exact and the epilogue is the same operations, so the outputs must be
the same bits as on packed codes and as those of slices of a few tokens, which run the weight-major kernel and, gated, the GEMV.
Shapes sit at the edges of its tiles: one k-block and odd counts of them (the last ring stage holds one), token
counts around the tile widths, weight rows past 64-, 128- and 256-row boundaries, tiles in several waves, K split into work
units, and gated layers from a few tokens.  With 8-bit codes the accumulators must be the oracle's integers."""

import numpy as np
import pytest
import torch

from oracle import qvla_oracle as O
from paper_2605_28803_gb300 import qvla as Q
from tests import gpu_helpers as G

pytestmark = pytest.mark.gpu

_T = {"f16": torch.float16, "bf16": torch.bfloat16}
_C = {"f16": Q.F16, "bf16": Q.BF16}


def _layer(rng, N, K, had, dt, gated=False):
    rows = 2 * N if gated else N
    wq = rng.integers(0, 256, (rows, K // 2), dtype=np.uint8)
    ws = (rng.uniform(0.5, 1.5, rows) / 64).astype(np.float32)
    bias = rng.standard_normal(rows).astype(np.float32)
    if gated:
        return Q.qvla_layer_create_gated(N, K, had, _C[dt], _C[dt], wq[:N], ws[:N], wq[N:], ws[N:], bias[:N], bias[N:]), wq
    return Q.qvla_layer_create(N, K, had, _C[dt], _C[dt], wq, ws, bias), wq


def _both(layer, x, M, dt):
    """The linear through its workspace, and the public halves on packed codes."""
    nb = Q.qvla_linear_workspace_bytes(layer, M)
    work = torch.full((nb,), 0xA5, dtype=torch.uint8, device=G.DEV)
    y = torch.full((M, layer.N), float("nan"), dtype=_T[dt], device=G.DEV)
    Q.qvla_linear_quantize(layer, x, M, -1, work, nb, G.stream())
    Q.qvla_linear_gemm(layer, work, nb, M, y, G.stream())
    xq = torch.empty(M, layer.K // 2, dtype=torch.uint8, device=G.DEV)
    xs = torch.empty(M, dtype=torch.float32, device=G.DEV)
    xsum = torch.empty(M, dtype=torch.int32, device=G.DEV)
    ref = torch.full((M, layer.N), float("nan"), dtype=_T[dt], device=G.DEV)
    Q.qvla_rotate_quantize(layer, x, M, -1, xq, xs, xsum, G.stream())
    Q.qvla_gemm_w4a4(layer, xq, xs, xsum, M, ref, None, G.stream())
    Q.qvla_check_device(G.stream())
    return y, ref


def _equal_slices(layer, x, y, rows):
    """The linear on slices of `rows` tokens, in other kernels, gives the same bits."""
    work = torch.empty(Q.qvla_linear_workspace_bytes(layer, rows), dtype=torch.uint8, device=G.DEV)
    for i in range(0, x.shape[0], rows):
        m = min(rows, x.shape[0] - i)
        part = torch.full((m, layer.N), float("nan"), dtype=y.dtype, device=G.DEV)
        Q.qvla_w4a4_linear(layer, x[i:], m, -1, part, work, work.numel(), G.stream())
        assert torch.equal(y[i : i + m], part)
    Q.qvla_check_device(G.stream())


@pytest.mark.parametrize("M,K,N,dt", [
    (129, 768, 16, "f16"), (160, 896, 272, "bf16"), (191, 1152, 528, "f16"), (192, 1024, 1040, "bf16"),
    (193, 2176, 1552, "f16"), (385, 1152, 4096, "bf16"), (2500, 1024, 2560, "f16"), (1500, 128, 4112, "bf16"),
    (150, 16384, 2048, "bf16"), (300, 16384, 2000, "f16"), (700, 16384, 1904, "bf16")])
def test_equals_the_other_kernels_bit_for_bit(M, K, N, dt):
    rng = np.random.default_rng(M * 7 + K + N)
    layer, _ = _layer(rng, N, K, 128, dt)
    x = torch.from_numpy(rng.standard_normal((M, K), dtype=np.float32)).to(_T[dt]).to(G.DEV)
    y, ref = _both(layer, x, M, dt)
    assert torch.equal(y, ref)
    _equal_slices(layer, x, y, 128)
    layer.close()


@pytest.mark.parametrize("M,K,H,dt", [(5, 128, 128, "bf16"), (33, 640, 256, "f16"), (128, 1152, 384, "bf16"),
                                      (130, 896, 384, "f16"), (816, 2048, 1024, "bf16"), (1000, 768, 8192, "f16")])
def test_gated_equals_packed_codes_and_slices(M, K, H, dt):
    rng = np.random.default_rng(M + K + H)
    layer, _ = _layer(rng, H, K, 64, dt, gated=True)
    x = torch.from_numpy(rng.standard_normal((M, K), dtype=np.float32)).to(_T[dt]).to(G.DEV)
    y, ref = _both(layer, x, M, dt)
    assert torch.equal(y, ref)
    _equal_slices(layer, x, y, 4)
    layer.close()


@pytest.mark.parametrize("M,K,N,gated,dt", [
    (129, 768, 16, False, "f16"), (150, 896, 512, False, "bf16"), (777, 4096, 1024, False, "f16"), (200, 16384, 2048, False, "bf16"),
    (500, 384, 528, False, "f16"), (2500, 1152, 2560, False, "bf16"), (4001, 1024, 4112, False, "f16"), (10, 1024, 2048, True, "bf16"),
    (50, 2176, 384, True, "f16"), (193, 1152, 1024, True, "bf16")])
def test_packed_codes_equal_slices_of_few_tokens(M, K, N, gated, dt):
    """Packed codes: the weight-major kernel (up to 128 tokens) and, for gated layers, the GEMV (4 tokens) on slices."""
    rng = np.random.default_rng(M + K + N)
    layer, _ = _layer(rng, N, K, 128, dt, gated)
    xq = torch.from_numpy(rng.integers(0, 256, (M, K // 2), dtype=np.uint8)).to(G.DEV)
    xq = torch.where((xq & 15) == 8, xq ^ 8, xq)  # codes -7 .. 7
    xq = torch.where((xq >> 4) == 8, xq ^ 0x80, xq)
    nib = torch.stack((xq & 15, xq >> 4), 2).to(torch.int32)
    xsum = ((nib ^ 8) - 8).sum((1, 2), dtype=torch.int32)
    xs = torch.from_numpy(rng.uniform(0.5, 1.5, M).astype(np.float32) / 64).to(G.DEV)
    y = torch.full((M, N), float("nan"), dtype=_T[dt], device=G.DEV)
    acc = torch.full((M, 2 * N if gated else N), -1, dtype=torch.int32, device=G.DEV)
    Q.qvla_gemm_w4a4(layer, xq, xs, xsum, M, y, acc, G.stream())
    rows = 4 if gated else 128
    for i in range(0, M, rows):
        m = min(rows, M - i)
        part = torch.empty(m, N, dtype=_T[dt], device=G.DEV)
        pacc = torch.empty(m, acc.shape[1], dtype=torch.int32, device=G.DEV)
        Q.qvla_gemm_w4a4(layer, xq[i : i + m].clone(), xs[i : i + m].clone(), xsum[i : i + m].clone(), m, part, pacc, G.stream())
        assert torch.equal(acc[i : i + m], pacc)
        assert torch.equal(y[i : i + m], part)
    Q.qvla_check_device(G.stream())
    layer.close()


@pytest.mark.parametrize("packed,M,K,N,gated", [
    (False, 485, 384, 19968, False), (False, 202, 896, 13312, False), (False, 199, 1152, 13056, False),
    (False, 131, 384, 21760, False), (False, 129, 1152, 21248, False), (False, 36, 384, 19968, True),
    (False, 33, 1152, 12288, True), (False, 99, 896, 10496, True), (False, 129, 896, 10496, True),
    (True, 195, 384, 19712, False), (True, 194, 1152, 20224, False), (True, 39, 384, 20480, True),
    (True, 34, 1664, 11264, True), (True, 99, 1152, 20224, True)])
def test_odd_k_blocks_over_several_tiles_a_pair(packed, M, K, N, gated):
    """An odd number of k-blocks leaves a tile's last ring stage half filled, and the next tile of the pair takes the same
    TMEM slots an odd number of stages later (3 at 128- and 160-token tiles, 5 at 64), from other converter warps.  Every run
    must be the bits of slices of a few tokens, on the weight-major kernel or, gated, the GEMV."""
    rng = np.random.default_rng(M + K + N)
    layer, _ = _layer(rng, N, K, 128, "f16", gated)
    y = torch.empty(M, N, dtype=torch.float16, device=G.DEV)
    if packed:
        q = rng.integers(-7, 8, (M, K)).astype(np.int8)
        xq = torch.from_numpy(O.pack_int4(q)).to(G.DEV)
        xsum = torch.from_numpy(q.sum(1, dtype=np.int32)).to(G.DEV)
        xs = torch.from_numpy(rng.uniform(0.5, 1.5, M).astype(np.float32) / 64).to(G.DEV)

        def run(i, m, out):
            Q.qvla_gemm_w4a4(layer, xq[i:], xs[i : i + m].clone(), xsum[i : i + m].clone(), m, out, None, G.stream())
    else:
        x = torch.from_numpy(rng.standard_normal((M, K), dtype=np.float32)).half().to(G.DEV)
        nb = Q.qvla_linear_workspace_bytes(layer, M)
        work = torch.empty(nb, dtype=torch.uint8, device=G.DEV)

        def run(i, m, out):
            Q.qvla_w4a4_linear(layer, x[i:], m, -1, out, work, nb, G.stream())

    rows = 4 if gated else 128
    want = torch.empty_like(y)
    for i in range(0, M, rows):
        run(i, min(rows, M - i), want[i:])
    for _ in range(20):
        y.fill_(float("nan"))
        run(0, M, y)
        assert torch.equal(y, want)
    Q.qvla_check_device(G.stream())
    layer.close()


@pytest.mark.parametrize("M,K,N,gated", [(200, 1152, 272, False), (129, 128, 16, False), (77, 896, 256, True)])
def test_eight_bit_codes_give_the_oracles_integers(M, K, N, gated):
    rng = np.random.default_rng(M + K)
    layer, wq = _layer(rng, N, K, 1, "f16", gated)
    xq = rng.integers(-127, 128, (M, K)).astype(np.int8)
    nb = Q.qvla_w4a8_workspace_bytes(layer, M)
    work = torch.empty(nb, dtype=torch.uint8, device=G.DEV)
    acc = torch.full((M, wq.shape[0]), -1, dtype=torch.int32, device=G.DEV)
    y = torch.empty(M, N, dtype=torch.float16, device=G.DEV)
    xs = torch.full((M,), 1e-4, dtype=torch.float32, device=G.DEV)
    Q.qvla_gemm_w4a8(layer, torch.from_numpy(xq).to(G.DEV), xs, M, y, acc, work, nb, G.stream())
    Q.qvla_check_device(G.stream())
    assert np.array_equal(acc.cpu().numpy(), O.int_gemm(xq, O.unpack_int4(wq)))
    layer.close()


def test_a_wait_that_runs_out_reports_timeout_and_the_next_launch_is_clean():
    """With the hook no copy is issued: every role's wait runs out, no MMA is issued, nothing is written, the kernel
    returns; the next launch is bit-exact."""
    rng = np.random.default_rng(3)
    M, K, N = 200, 1024, 512
    layer, _ = _layer(rng, N, K, 128, "f16")
    x = torch.from_numpy(rng.standard_normal((M, K), dtype=np.float32)).half().to(G.DEV)
    y0, ref = _both(layer, x, M, "f16")
    assert torch.equal(y0, ref)
    nb = Q.qvla_linear_workspace_bytes(layer, M)
    work = torch.empty(nb, dtype=torch.uint8, device=G.DEV)
    y = torch.full((M, N), float("nan"), dtype=torch.float16, device=G.DEV)
    Q.qvla_debug_set_hooks(20_000_000, True)
    try:
        Q.qvla_w4a4_linear(layer, x, M, -1, y, work, nb, G.stream())
        with pytest.raises(Q.QvlaError) as e:
            Q.qvla_check_device(G.stream())
        assert e.value.status == 6
        assert torch.isnan(y).all().item()
    finally:
        Q.qvla_debug_set_hooks(0, False)
    Q.qvla_check_device(G.stream())
    y1, _ = _both(layer, x, M, "f16")
    assert torch.equal(y1, y0)
    layer.close()
