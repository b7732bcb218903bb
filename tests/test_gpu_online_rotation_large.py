"""GPU parity of the online rotation's two kernels for large batches (csrc/block_rotate.cu; Sec. 4.1 Eq. 4-5): a pass that
permutes rows, then the blocks in place.  They sum in the order of the kernel for small batches, so the same rows in slices
below the line give the same bits.  Odd row counts (the permutation takes 16-bit rows in pairs), a last tile of one row, row
widths off every stride, infinities and NaN; a pointer that is not 16-byte aligned stays on the small batches' kernel."""

import numpy as np
import pytest
import torch

from paper_2605_28803_gb300 import qvla as Q
from tests import gpu_helpers as G

pytestmark = pytest.mark.gpu


def _layer(K, block, dt):
    rng = np.random.default_rng(K + block)
    layer = Q.qvla_layer_create(16, K, 128, Q.DTYPE_CODES[dt], Q.F16, np.zeros((16, K // 2), np.uint8),
                                np.ones(16, np.float32), None)
    Q.qvla_layer_set_online_rotation(layer, rng.permutation(K).astype(np.int32),
                                     rng.standard_normal((K // block, block, block)).astype(np.float32), block)
    return layer


def _rotate(layer, x, out):
    Q.qvla_online_rotate(layer, x, x.shape[0], out, G.stream())
    Q.qvla_check_device(G.stream())
    return out


@pytest.mark.parametrize("dt", ["f16", "bf16", "f32"])
@pytest.mark.parametrize("M,K,block", [(2048, 1024, 64), (2049, 1024, 16), (1153, 2944, 32), (129, 16384, 64), (1025, 2176, 64),
                                       (171, 12288, 32)])
def test_large_batches_equal_slices(dt, M, K, block):
    t = {"f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}[dt]
    layer = _layer(K, block, dt)
    g = torch.Generator().manual_seed(M)
    x = torch.randn(M, K, generator=g)
    x[3, 5], x[7, K - 1], x[M - 1, 0] = np.inf, np.nan, -np.inf
    x = x.to(t).to(G.DEV)
    got = _rotate(layer, x, torch.full_like(x, 3.0))
    rows = 120
    want = torch.cat([_rotate(layer, x[i : i + rows].contiguous(), torch.empty_like(x[i : i + rows])) for i in range(0, M, rows)])
    bits = torch.int32 if dt == "f32" else torch.int16
    same = (got.view(bits) == want.view(bits)) | (got.isnan() & want.isnan())
    assert bool(same.all())
    shifted = torch.empty(M * K + 1, dtype=t, device=G.DEV)
    out = _rotate(layer, x, shifted[1:].view(M, K))
    assert bool(((out == got) | (got.isnan() & out.isnan())).all())
    layer.close()
