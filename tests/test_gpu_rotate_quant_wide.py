"""GPU parity of the rotate-quantise kernel with 32 channels per thread (csrc/rotate_quant_wide.cuh; Sec. 4.1 Eq. 3-5,
Sec. 4.2 Eq. 5-6).

It takes 4-bit codes with one scale per row, but for a few long rows, which the pass kernel keeps (at most 48 rows of more
than 4096 channels; its codes, scales and sums are pinned elsewhere).  A row repeated r times side by side has the same
rotated values, the same maximum and r times the code sum, so the pass kernel on repeated rows pins this one at every
width.  A per-group table of equal scales takes the 64-channel kernel for groups of 2048 and 4096 channels, which pins the
per-step codes of such blocks, and this kernel for smaller groups, whose codes and sums equal those of the groups taken as rows
of their own.  Blocks at every phase count and group size, row widths that are not a power of two of threads, ragged rows per
CTA, per token and per step with clamping, exact ties, zero rows, huge, tiny, infinite and NaN values."""

import numpy as np
import pytest
import torch

from paper_2605_28803_gb300 import qvla as Q
from tests import gpu_helpers as G

pytestmark = pytest.mark.gpu

_T = {"f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}


def _quantise(layer, x, step=-1):
    M, K = x.shape
    nb = Q.qvla_linear_workspace_bytes(layer, M)
    work = torch.full((nb,), 0x3C, dtype=torch.uint8, device=G.DEV)
    Q.qvla_linear_quantize(layer, x.contiguous(), M, step, work, nb, G.stream())
    Q.qvla_check_device(G.stream())
    r256 = lambda v: (v + 255) // 256 * 256  # noqa: E731
    o = r256(M * K)
    return (work[: M * K].view(M, K).cpu(), work[o : o + 4 * M].view(torch.int32).cpu(),
            work[o + r256(4 * M) : o + r256(4 * M) + 4 * M].view(torch.int32).cpu())


def _packed(x, had, scale=None):
    M, K = x.shape
    xq = torch.full((M, K // 2), 0x3C, dtype=torch.uint8, device=G.DEV)
    xs = torch.empty(M, dtype=torch.float32, device=G.DEV)
    xsum = torch.empty(M, dtype=torch.int32, device=G.DEV)
    code = {torch.float16: Q.F16, torch.bfloat16: Q.BF16, torch.float32: Q.F32}[x.dtype]
    Q.qvla_rotate_quantize_rows(x.contiguous(), code, M, K, had, scale, xq, xs, xsum, G.stream())
    Q.qvla_check_device(G.stream())
    return xq.cpu(), xs.view(torch.int32).cpu(), xsum.cpu()


def _unpack(xq):
    """Packed nibbles -> operand bytes q + 8 in the order k0 k2 k4 k6 k1 k3 k5 k7."""
    M, K2 = xq.shape
    c = torch.stack((xq & 15, xq >> 4), 2).view(M, K2 // 4, 8) ^ 8
    return torch.cat((c[:, :, 0::2], c[:, :, 1::2]), 2).reshape(M, 2 * K2)


def _values(rng, M, K, had, dt, special=True):
    x = rng.standard_normal((M, K)).astype(np.float32)
    x[:, rng.choice(K, max(1, K // 200), replace=False)] *= 20.0
    if special and M > 8:
        x[1] = 0.0
        x[2] *= 1e-6 if dt == "f16" else 1e-38
        x[3, 5] = 6e4 if dt == "f16" else 1e38
        x[4, 7] = np.inf
        x[5, K - 1] = np.nan
        x[6] = np.where(rng.random(K) < 0.5, 7.0, np.round(rng.uniform(-7, 7, K) * 2) / 2)  # ties where had = 1
        x[7, 0], x[7, 1:] = 1.0, 0.0  # one channel: every rotated value equal
    return torch.from_numpy(x).to(_T[dt]).to(G.DEV)


@pytest.mark.parametrize("M,K,had,dt,r", [
    (65, 128, 128, "f16", 64), (70, 384, 32, "bf16", 16), (131, 256, 64, "f16", 32), (130, 768, 256, "bf16", 8),
    (129, 512, 512, "bf16", 16), (66, 2560, 512, "f16", 4), (100, 1024, 1024, "bf16", 8), (97, 3072, 1024, "f16", 4),
    (130, 2048, 2048, "bf16", 4), (70, 6144, 2048, "f16", 1), (66, 16384, 2048, "bf16", 1), (200, 640, 1, "f16", 16),
    (66, 4096, 16, "bf16", 2), (9, 2048, 256, "f16", 4), (50, 1024, 64, "bf16", 8),
    (77, 640, 128, "bf16", 16), (300, 896, 64, "f16", 16)])
def test_a_batch_equals_the_pass_kernel_on_repeated_rows(M, K, had, dt, r):
    rng = np.random.default_rng(M + K + had)
    x = _values(rng, M, K, had, dt)
    xr = x.repeat(1, r)
    make = lambda k: Q.qvla_layer_create(16, k, had, Q.DTYPE_CODES[dt], Q.F16, np.zeros((16, k // 2), np.uint8),  # noqa: E731
                                         np.ones(16, np.float32), None)
    layer, wide = make(K), make(K * r)
    table = np.array([0.31, 1.7e-3, 3e-39], np.float32)  # an ordinary scale, one that clamps, an overflowing reciprocal
    Q.qvla_set_step_scales(layer, table)
    Q.qvla_set_step_scales(wide, table)
    for step in (-1, 0, 1, 2):
        ob, xs, xsum = _quantise(layer, x, step)
        parts = [_quantise(wide, xr[i : i + 48], step) for i in range(0, M, 48)] if r > 1 or M > 48 else []
        want = [torch.cat(p) for p in zip(*parts)]
        assert torch.equal(ob.repeat(1, r), want[0])
        assert torch.equal(xs, want[1]) and torch.equal(r * xsum, want[2])
        scale = None if step < 0 else torch.tensor([table[step]], device=G.DEV)
        xq, pxs, pxsum = _packed(x, had, scale)
        assert torch.equal(_unpack(xq), ob) and torch.equal(pxs, xs) and torch.equal(pxsum, xsum)
    layer.close()
    wide.close()


@pytest.mark.parametrize("xdt,ydt", [("bf16", "bf16"), ("f16", "f16"), ("f32", "f16")])
@pytest.mark.parametrize("K,had", [(128, 1), (640, 128), (2048, 2048), (4096, 16), (4096, 4096), (6144, 2048), (16384, 1), (16384, 2048)])
def test_a_nan_token_gives_a_nan_row(K, had, xdt, ydt):
    """One NaN channel of a token under a scale per token makes its scale NaN and its outputs NaN, on every kernel that
    quantises (one launch at one token, the passes, 32 channels a thread, 8-bit codes); the other tokens' outputs stay."""
    rng = np.random.default_rng(K + had)
    N = 32
    layer = Q.qvla_layer_create(N, K, had, Q.DTYPE_CODES[xdt], Q.DTYPE_CODES[ydt], rng.integers(0, 256, (N, K // 2), dtype=np.uint8),
                                np.full(N, 1e-3, np.float32), rng.standard_normal(N).astype(np.float32))
    for M in (1, 2, 4, 33, 50, 64, 65, 200):
        x = torch.from_numpy(rng.standard_normal((M, K)).astype(np.float32)).to(_T[xdt]).to(G.DEV)
        bad = x.clone()
        bad[M // 2, int(rng.integers(K))] = np.nan
        nb = max(Q.qvla_linear_workspace_bytes(layer, M), Q.qvla_w4a8_workspace_bytes(layer, M))
        work = torch.empty(nb, dtype=torch.uint8, device=G.DEV)
        for linear in (Q.qvla_w4a4_linear,) + ((Q.qvla_w4a8_linear,) if K <= 4096 else ()):
            y, want = (torch.zeros(M, N, dtype=_T[ydt], device=G.DEV) for _ in range(2))
            linear(layer, bad, M, -1, y, work, nb, G.stream())
            linear(layer, x, M, -1, want, work, nb, G.stream())
            Q.qvla_check_device(G.stream())
            want[M // 2] = np.nan
            assert torch.equal(y.isnan(), want.isnan())
            assert torch.equal(y[~y.isnan()], want[~want.isnan()])
    layer.close()


def _graph_us(call, n=10):
    """Least time of a call among n back to back in a graph, over 12 replays."""
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        call(s)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            for _ in range(n):
                call(s)
        best = float("inf")
        for _ in range(12):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record(s)
            g.replay()
            b.record(s)
            s.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3 / n)
    return best


@pytest.mark.parametrize("M,K,had,dt", [(3200, 16384, 2048, "f16"), (3325, 10112, 128, "bf16")])
def test_rows_of_zeros_cost_no_more_than_others(M, K, had, dt):
    """Padding tokens stay on the fast path: as fast as other rows (a tenth allowed for the timing; the path that decides every
    code exactly takes 1.28 and 1.34 times as long on these shapes).  Their codes, scales and sums are 0."""
    xq = torch.full((M, K // 2), 0x3C, dtype=torch.uint8, device=G.DEV)
    xs = torch.ones(M, dtype=torch.float32, device=G.DEV)
    xsum = torch.ones(M, dtype=torch.int32, device=G.DEV)
    x = torch.randn(M, K, device=G.DEV).to(_T[dt])
    us = []
    for v in (x, torch.zeros_like(x)):
        us.append(_graph_us(lambda s: Q.qvla_rotate_quantize_rows(v, Q.DTYPE_CODES[dt], M, K, had, None, xq, xs, xsum, s)))
    assert not xq.any() and not xs.any() and not xsum.any()
    assert us[1] <= 1.1 * us[0], us


@pytest.mark.parametrize("M,K,had", [(67, 2304, 256), (131, 1024, 1024), (70, 4096, 2048), (65, 384, 32), (33, 8192, 4096),
                                      (33, 2944, 128), (40, 10112, 64), (50, 12288, 4096)])
def test_f32_rows_equal_bf16_rows_of_the_same_values(M, K, had):
    rng = np.random.default_rng(K)
    xb = _values(rng, M, K, had, "bf16")
    for got, want in zip(_packed(xb.float(), had), _packed(xb, had)):
        assert torch.equal(got, want)


@pytest.mark.parametrize("M,K,had", [(80, 1024, 64), (66, 2048, 128), (130, 4096, 2048), (1, 4096, 4096),
                                      (66, 8192, 4096), (50, 4096, 4096), (142, 2944, 64), (70, 10112, 128), (500, 384, 128)])
def test_step_codes_equal_the_64_channel_kernel(M, K, had):
    """A per-group table of one repeated scale runs the 64-channel kernel from groups of 2048: the same outputs follow."""
    rng = np.random.default_rng(K + had)
    x = _values(rng, M, K, had, "f16", special=False)
    wq = rng.integers(0, 256, (32, K // 2), dtype=np.uint8)
    ws = np.full(32, 2.0 ** -8, np.float32)
    out = []
    for grouped in (False, True):
        layer = Q.qvla_layer_create(32, K, had, Q.F16, Q.F16, wq, ws, None)
        if grouped:
            Q.qvla_set_step_group_scales(layer, np.full((1, K // max(128, had)), 0.25, np.float32))
        else:
            Q.qvla_set_step_scales(layer, np.array([0.25], np.float32))
        nb = Q.qvla_linear_workspace_bytes(layer, M)
        work = torch.empty(nb, dtype=torch.uint8, device=G.DEV)
        y = torch.empty(M, 32, dtype=torch.float16, device=G.DEV)
        Q.qvla_w4a4_linear(layer, x, M, 0, y, work, nb, G.stream())
        Q.qvla_check_device(G.stream())
        out.append(work[: M * K].cpu())
        layer.close()
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("M,K,had,dt", [(50, 1024, 64, "f16"), (142, 2944, 128, "bf16"), (700, 384, 1, "f16"), (33, 2560, 512, "bf16"),
                                         (65, 3072, 1024, "f16"), (9, 512, 256, "bf16"), (3000, 256, 32, "f16")])
def test_group_codes_equal_the_groups_as_rows(M, K, had, dt):
    rng = np.random.default_rng(M + K)
    x = _values(rng, M, K, had, dt, special=False)
    group = max(128, had)
    n = K // group
    table = rng.uniform(0.05, 0.6, n).astype(np.float32)
    layer = Q.qvla_layer_create(16, K, had, Q.DTYPE_CODES[dt], Q.F16, np.zeros((16, K // 2), np.uint8), np.ones(16, np.float32), None)
    Q.qvla_set_step_group_scales(layer, table[None, :])
    nb = Q.qvla_linear_workspace_bytes(layer, M)
    work = torch.full((nb,), 0x3C, dtype=torch.uint8, device=G.DEV)
    y = torch.empty(M, 16, dtype=torch.float16, device=G.DEV)
    Q.qvla_w4a4_linear(layer, x, M, 0, y, work, nb, G.stream())
    Q.qvla_check_device(G.stream())
    r256 = lambda v: (v + 255) // 256 * 256  # noqa: E731
    codes = work[: M * K].view(M, n, group).cpu()
    o = r256(M * K) + 2 * r256(4 * M)
    gsum = work[o : o + 4 * M * n].view(torch.int32).view(M, n).cpu()
    part = Q.qvla_layer_create(16, group, had, Q.DTYPE_CODES[dt], Q.F16, np.zeros((16, group // 2), np.uint8), np.ones(16, np.float32),
                               None)
    Q.qvla_set_step_scales(part, table)
    for g in range(n):
        ob, _, xsum = _quantise(part, x[:, g * group : (g + 1) * group], g)
        assert torch.equal(codes[:, g], ob) and torch.equal(gsum[:, g], xsum)
    part.close()
    layer.close()


@pytest.mark.parametrize("K", range(128, 16385, 128))
def test_every_row_width_runs(K):
    """Every K, with many rows a CTA and one: the shared memory and thread counts of each width are accepted, and a
    row's code sum is that of its codes."""
    x = torch.randn(153 if K % 256 else 80, K, device=G.DEV, dtype=torch.float16)
    xq, _, xsum = _packed(x, 64)
    codes = _unpack(xq).to(torch.int32) - 8
    assert torch.equal(codes.sum(1, dtype=torch.int32), xsum)
    assert int(codes.abs().max()) == 7


@pytest.mark.parametrize("M,K,log_b,dt", [(m, k, b, d) for b, (m, k, d) in enumerate([
    (200, 640, "f16"), (33, 128, "bf16"), (70, 384, "f32"), (5, 1152, "f16"), (300, 256, "bf16"), (9, 3200, "f16"),
    (77, 2944, "bf16"), (129, 896, "f16"), (50, 2304, "f32"), (65, 1536, "f16"), (8, 3072, "bf16"), (130, 2048, "f16"),
    (50, 4096, "bf16")])])
def test_eight_bit_codes_of_every_block(M, K, log_b, dt):
    """Codes within half a step of the float64 rotation (a float32 rotation's error of a step's 2^-9 added), code sums theirs, and the
    linear's operand planes equal those made from the int8 rows (the same outputs)."""
    had = 1 << log_b
    rng = np.random.default_rng(K + log_b)
    x = _values(rng, M, K, had, dt, special=False)
    code = Q.DTYPE_CODES[dt]
    xq = torch.full((M, K), 99, dtype=torch.int8, device=G.DEV)
    xs = torch.empty(M, dtype=torch.float32, device=G.DEV)
    xsum = torch.empty(M, dtype=torch.int32, device=G.DEV)
    Q.qvla_rotate_quantize_rows_a8(x, code, M, K, had, None, xq, xs, xsum, G.stream())
    h = torch.ones(1, 1, dtype=torch.float64)
    for _ in range(log_b):
        h = torch.cat((torch.cat((h, h), 1), torch.cat((h, -h), 1)), 0)
    z = (x.double().cpu().view(M, K // had, had) @ (h / had ** 0.5)).reshape(M, K)
    step = z.abs().amax(1) / 127
    assert torch.allclose(xs.double().cpu(), step, rtol=1e-5, atol=0)
    q = xq.cpu().double()
    assert float((q - z / step[:, None]).abs().max()) <= 0.5 + 2.0 ** -9
    assert torch.equal(xq.to(torch.int32).sum(1, dtype=torch.int32), xsum)
    layer = Q.qvla_layer_create(32, K, had, code, Q.F16, rng.integers(0, 256, (32, K // 2), dtype=np.uint8),
                                np.full(32, 1e-3, np.float32), None)
    nb = Q.qvla_w4a8_workspace_bytes(layer, M)
    work = torch.empty(nb, dtype=torch.uint8, device=G.DEV)
    y, want = (torch.empty(M, 32, dtype=torch.float16, device=G.DEV) for _ in range(2))
    Q.qvla_w4a8_linear(layer, x, M, -1, y, work, nb, G.stream())
    Q.qvla_gemm_w4a8(layer, xq, xs, M, want, None, work, nb, G.stream())
    Q.qvla_check_device(G.stream())
    assert torch.equal(y, want)
    layer.close()
