"""The cases whose speed is measured: calls of libqvla's public entry points (the ctypes binding and the stack
runner) on synthetic data of the backbone's and the action head's shapes, from one 512-wide layer to batches of
8192 tokens.

A case is a dict of plain values:
  kind   "linear"  one qvla_w4a4_linear (options: gated, a per-step table, a bias, an online rotation)
         "grouped" one qvla_w4a4_linear with a per-step table of one scale per channel group
         "a8"      one qvla_w4a8_linear (8-bit activation codes)
         "codes"   qvla_rotate_quantize_rows, then qvla_gemm_w4a4 on the packed codes
         "mlp"     the gated MLP: the gate/up linear, then the down linear on its output
         "stack"   LinearStack: a sequence of linears captured once as a CUDA graph and replayed
  m, k, n, had     tokens, input channels, output channels (hidden units when gated), Hadamard block
  x, y             input and output types

Weights are int4 codes of Gaussian weights with a float32 scale per output channel; activations are N(0, 1) with 0.5 %
of the channels 20 times larger (the action head's: N(0, sigma^2) of a denoising step).  `exact` is the float64
statement of the method in plain torch: block Hadamard, scale, round half to even, integer product, dequantisation;
values that pass from one call to the next are rounded to the type they are passed in.
"""

import math

import torch

from paper_2605_28803_gb300 import qvla as Q
from paper_2605_28803_gb300.stack import LinearStack
from paper_2605_28803_gb300.workloads import StackWeights

DEV = "cuda"
_TORCH = {"f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}
_CODE = {"f16": Q.F16, "bf16": Q.BF16, "f32": Q.F32}

# (K, N, gated) of one block of the action head and of one layer of the backbone, as run
DIT_BLOCK = ((1024, 3072, False), (1024, 1024, False), (1024, 4096, False), (4096, 1024, False))
BACKBONE_LAYER = ((2048, 2560, False), (2048, 2048, False), (2048, 16384, True), (16384, 2048, False))


def listed():
    return [
        # the smallest layer of the test configurations: 64 tokens, 512 -> 512, one scale of a 10-step table
        dict(name="layer_64x512", kind="linear", m=64, k=512, n=512, had=512, x="f16", y="f16", gated=False, step=True,
             bias=False, rot=0),
        # decoding one token: two layers of the backbone (8 linears) as one graph
        dict(name="backbone_decode", kind="stack", shapes="backbone", layers=2, m=1, x="bf16", step=False),
        # a small batch of decode tokens through the widest reduction
        dict(name="down_16", kind="linear", m=16, k=16384, n=2048, had=2048, x="bf16", y="bf16", gated=False, step=False,
             bias=False, rot=0),
        # one denoising step of the action head: 50 action tokens, 6 blocks (24 linears) as one graph
        dict(name="dit_step", kind="stack", shapes="dit", layers=6, m=50, x="f16", step=True),
        # the same head's up projection with one scale per step and 128-channel group, rotation blocks of 64
        dict(name="dit_grouped", kind="grouped", m=50, k=1024, n=4096, had=64, x="f16", y="f16"),
        # an odd layer and batch: 201 tokens, 9 Hadamard blocks, a weight count off every tile
        dict(name="odd_201", kind="linear", m=201, k=2304, n=1552, had=256, x="f16", y="f16", gated=False, step=True,
             bias=True, rot=0),
        # prefill: the backbone's gated MLP over a prefix of 816 tokens
        dict(name="mlp_816", kind="mlp", m=816, k=2048, n=16384, had=2048, x="bf16"),
        # prefill: a projection whose rotation P.U cannot be folded upstream and runs online
        dict(name="online_816", kind="linear", m=816, k=2048, n=2560, had=2048, x="bf16", y="bf16", gated=False,
             step=False, bias=False, rot=64),
        # 8-bit activation codes, the gate/up projection of the backbone
        dict(name="a8_gate_up_816", kind="a8", m=816, k=2048, n=16384, had=2048, x="bf16", y="bf16", gated=True,
             step=False),
        # the two halves through the public packed codes, float32 activations, an odd number of tokens
        dict(name="codes_777", kind="codes", m=777, k=4096, n=1024, had=4096, x="f32", y="f16"),
        # many requests at once: 64 action chunks of 50 tokens, the widest reduction
        dict(name="down_3200", kind="linear", m=3200, k=16384, n=2048, had=2048, x="f16", y="f16", gated=False, step=False,
             bias=False, rot=0),
        # the largest batch of the sweep
        dict(name="wide_8192", kind="linear", m=8192, k=2048, n=16384, had=2048, x="f16", y="f16", gated=False, step=False,
             bias=False, rot=0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _hadamard(rng, k, most=4096):
    """The largest power of two that divides K (the default), or the paper's block of 64."""
    b = 1
    while b < most and k % (2 * b) == 0:
        b *= 2
    return b if rng.random() < 0.7 else min(b, 64)


def draw(rng):
    while True:
        kind = rng.choice(["linear", "linear", "linear", "mlp", "stack", "grouped", "a8", "codes"])
        k = 128 * round(_log(rng, 2, 128))
        n = 16 * round(_log(rng, 8, 1024))
        m = round(_log(rng, 1, 8192))
        x = rng.choice(["f16", "bf16"])
        c = dict(kind=kind, m=m, k=k, n=n, had=_hadamard(rng, k), x=x, y=x)
        if kind == "linear":
            c.update(gated=rng.random() < 0.25, step=rng.random() < 0.4, bias=rng.random() < 0.4,
                     rot=rng.choice([0, 0, 0, 0, 16, 32, 64]))
            if rng.random() < 0.1:
                c["x"] = "f32"
        elif kind == "grouped":
            c["had"] = 64
        elif kind == "a8":
            c["k"] = k = min(k, 4096)
            c.update(gated=rng.random() < 0.5, step=rng.random() < 0.4, had=_hadamard(rng, k))
        elif kind == "codes":
            c["x"] = rng.choice(["f16", "bf16", "f32"])
        elif kind == "mlp":
            c["k"] = k = 128 * round(_log(rng, 2, 16))
            c["had"] = _hadamard(rng, k, 2048)
            del c["y"]
        elif kind == "stack":
            dit = rng.random() < 0.5
            c = dict(kind=kind, shapes="dit" if dit else "backbone", layers=rng.randint(1, 6 if dit else 2),
                     m=round(_log(rng, 8, 300) if dit else _log(rng, 1, 300)), x="f16" if dit else "bf16", step=dit)
        if c.get("gated") or kind == "mlp":
            c["n"] = max(128, c["n"] // 128 * 128)
        w = work(c)
        if w["flops"] <= 5.4e11 and w["bytes"] <= 3.1e8 and _weights(c) <= 7e7:
            return c


# ---- shapes -------------------------------------------------------------------------------------------------------

def _linears(case):
    """(k, n, gated, had, bias) of every linear of the case."""
    if case["kind"] == "stack":
        if case["shapes"] == "dit":
            return [(k, n, g, k, True) for k, n, g in DIT_BLOCK] * case["layers"]
        return [(k, n, g, min(k, 2048), False) for k, n, g in BACKBONE_LAYER] * case["layers"]
    if case["kind"] == "mlp":
        return [(case["k"], case["n"], True, case["had"], False), (case["n"], case["k"], False, _wide(case["n"]), False)]
    return [(case["k"], case["n"], case.get("gated", False), case["had"], case.get("bias", False))]


def _wide(k):
    """The Hadamard block of the MLP's hidden units."""
    b = 1
    while b < 2048 and k % (2 * b) == 0:
        b *= 2
    return b


def _weights(case):
    return sum(k * n * (2 if g else 1) for k, n, g, _, _ in _linears(case))


def work(case):
    size = {"f16": 2, "bf16": 2, "f32": 4}
    m, nbytes, flops = case["m"], 0, 0
    for i, (k, n, g, _, bias) in enumerate(_linears(case)):
        rows = 2 * n if g else n
        nbytes += rows * k // 2 + (8 if bias else 4) * rows  # codes, scales and biases
        nbytes += 2 * m * n
        if not (case["kind"] == "mlp" and i == 1):  # the MLP's hidden units are its own
            nbytes += m * k * size[case["x"]]
        flops += 2 * m * k * rows
        if case.get("rot"):
            nbytes += k * case["rot"] * 4
            flops += 2 * m * k * case["rot"]
    if case["kind"] == "codes":  # the packed codes, scales and sums are outputs too
        nbytes += m * case["k"] // 2 + 8 * m
    return {"bytes": nbytes, "flops": flops}


# ---- inputs -------------------------------------------------------------------------------------------------------

class _Inputs:
    """Everything a case is drawn from, in a fixed order from one generator."""

    def __init__(self, case, seed):
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        self.case, self.layers = case, []
        m, x = case["m"], _TORCH[case["x"]]
        dit = case.get("shapes") == "dit"
        for i, (k, n, gated, had, bias) in enumerate(_linears(case)):
            rows = 2 * n if gated else n
            codes = torch.randn(rows, k, generator=g, device=DEV).mul_(2.0).round_().clamp_(-7, 7).to(torch.int8)
            scale = (0.8 + 0.4 * torch.rand(rows, generator=g, device=DEV)) * (0.5 / math.sqrt(k))
            b = 0.05 * torch.randn(rows, generator=g, device=DEV) if bias else None
            self.layers.append((k, n, gated, had, codes, scale, b))
        self.x = []
        for i, layer in enumerate(self.layers):
            if case["kind"] == "mlp" and i == 1:
                break
            k = layer[0]
            v = torch.randn(m, k, generator=g, device=DEV)
            if dit or case["kind"] == "grouped":
                v *= 4.0 * 0.125 ** (3 / 9)  # the fourth of ten denoising steps
                if case["kind"] == "grouped":  # uneven channels, what per-group scales are for
                    prof = torch.exp(0.8 * torch.randn((k + 63) // 64, generator=g, device=DEV))
                    v *= prof.repeat_interleave(64)[None, :k]
            else:
                idx = torch.randperm(k, generator=g, device=DEV)[: max(1, round(0.005 * k))]
                v[:, idx] *= 20.0
            self.x.append(v.to(x))
        # per-step tables: the peak of the rotated activations of other tokens, over the largest code
        self.tables = None
        if case.get("step") or case["kind"] == "grouped":
            qmax = 127.0 if case["kind"] == "a8" else 7.0
            self.tables = []
            for layer, v in zip(self.layers, self.x):
                k, had = layer[0], layer[3]
                cal = v[torch.randperm(m, generator=g, device=DEV)[:16]].double()
                peak = _fwht(cal, had).abs().amax(0)
                if case["kind"] == "grouped":
                    peak = peak.view(-1, max(128, had)).amax(1)
                else:
                    peak = peak.amax().view(1)
                grow = 1.0 + 0.1 * torch.arange(10, dtype=torch.float64, device=DEV)
                self.tables.append((grow[:, None] * peak[None, :] / qmax).float())
        self.perm = self.rot = None
        if case.get("rot"):
            k, blk = self.layers[0][0], case["rot"]
            self.perm = torch.randperm(k, generator=g, device=DEV).to(torch.int32)
            a = torch.randn(k // blk, blk, blk, generator=g, device=DEV, dtype=torch.float32).double().cpu()
            self.rot = torch.linalg.qr(a)[0].contiguous()


STEP = 3  # the row of the table that a pass uses


def _pack(codes):
    u = codes.to(torch.int16).bitwise_and(15).to(torch.uint8)
    return (u[:, 0::2] | (u[:, 1::2] << 4)).contiguous().cpu().numpy()


def _cpu(t):
    return None if t is None else t.cpu().numpy()


def _layer(layer, xdt, ydt):
    k, n, gated, had, codes, scale, bias = layer
    wq, ws, b = _pack(codes), _cpu(scale), _cpu(bias)
    if not gated:
        return Q.qvla_layer_create(n, k, had, xdt, ydt, wq, ws, b)
    return Q.qvla_layer_create_gated(n, k, had, xdt, ydt, wq[:n], ws[:n], wq[n:], ws[n:],
                                     None if b is None else b[:n], None if b is None else b[n:])


def prepare(case, seed):
    """The program's layers (with their tables and rotations), workspace and buffers."""
    inp = _Inputs(case, seed)
    kind, m = case["kind"], case["m"]
    if kind == "stack":
        weights = [StackWeights(str(i), k, n, had, _pack(codes), _cpu(scale), _cpu(bias), gated=gated)
                   for i, (k, n, gated, had, codes, scale, bias) in enumerate(inp.layers)]
        stack = LinearStack(weights, m, case["x"], case["x"])
        for i, v in enumerate(inp.x):
            stack.set_input(i, v)
        if inp.tables:
            stack.set_step_tables([_cpu(t[:, 0]) for t in inp.tables])
        return {"kind": kind, "stack": stack, "graph": stack.capture(STEP if inp.tables else -1)}
    xdt = _CODE[case["x"]]
    ydt = _CODE[case.get("y", case["x"])]
    layers = [_layer(v, xdt, ydt) for v in inp.layers]
    s = {"kind": kind, "m": m, "x": inp.x[0], "layers": layers, "step": STEP if inp.tables else -1}
    if kind == "grouped":
        Q.qvla_set_step_group_scales(layers[0], _cpu(inp.tables[0]))
    elif inp.tables:
        Q.qvla_set_step_scales(layers[0], _cpu(inp.tables[0][:, 0]))
    if inp.rot is not None:
        Q.qvla_layer_set_online_rotation(layers[0], _cpu(inp.perm), inp.rot.numpy(), case["rot"])
    if kind == "codes":
        k = case["k"]
        s.update(xdt=xdt, k=k, had=case["had"], xq=torch.empty(m, k // 2, dtype=torch.uint8, device=DEV),
                 xscale=torch.empty(m, dtype=torch.float32, device=DEV),
                 xsum=torch.empty(m, dtype=torch.int32, device=DEV))
    else:
        nbytes = Q.qvla_w4a8_workspace_bytes if kind == "a8" else Q.qvla_linear_workspace_bytes
        s["wbytes"] = max(nbytes(layer, m) for layer in layers)
        s["work"] = torch.empty(s["wbytes"], dtype=torch.uint8, device=DEV)
    s["y"] = [torch.empty(m, layer.N, dtype=_TORCH[case.get("y", case["x"])], device=DEV) for layer in layers]
    return s


def run(s):
    kind = s["kind"]
    if kind == "stack":
        s["graph"].replay()
        return list(s["stack"].y)
    stream = torch.cuda.current_stream()
    m, layers, y = s["m"], s["layers"], s["y"]
    if kind == "codes":
        Q.qvla_rotate_quantize_rows(s["x"], s["xdt"], m, s["k"], s["had"], None, s["xq"], s["xscale"], s["xsum"], stream)
        Q.qvla_gemm_w4a4(layers[0], s["xq"], s["xscale"], s["xsum"], m, y[0], None, stream)
        return {"codes": s["xq"], "scale": s["xscale"], "sum": s["xsum"], "y": y[0]}
    linear = Q.qvla_w4a8_linear if kind == "a8" else Q.qvla_w4a4_linear
    linear(layers[0], s["x"], m, s["step"], y[0], s["work"], s["wbytes"], stream)
    if kind == "mlp":
        linear(layers[1], y[0], m, s["step"], y[1], s["work"], s["wbytes"], stream)
    return y


# ---- float64 statement of the method ------------------------------------------------------------------------------

def _fwht(x, b):
    """Normalised block Walsh-Hadamard transform along the rows (natural order)."""
    m, k = x.shape
    h = 1
    while h < b:
        v = x.view(m, k // (2 * h), 2, h)
        x = torch.stack((v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]), 2).view(m, k)
        h *= 2
    return x / math.sqrt(b)


def _quantise(x, had, table, qmax):
    """(codes, scales): the scale per row, the step's, or the step's per channel group."""
    z = _fwht(x.double(), had)
    if table is None:
        delta = z.abs().amax(1, keepdim=True) / qmax
    else:
        t = table[STEP].double()
        delta = t.repeat_interleave(z.shape[1] // t.numel())[None, :]
    return (z / delta).round().clamp(-qmax, qmax), delta


def _product(q, delta, layer):
    k, n, gated, had, codes, scale, bias = layer
    y = (q * delta) @ codes.double().t() * scale.double()
    if bias is not None:
        y = y + bias.double()
    return y


def _glue(y, n, dtype):
    """h = gelu(gate) * up of the gate and up outputs rounded to the output type."""
    gate, up = (v.to(dtype).double() for v in (y[:, :n], y[:, n:]))
    return torch.nn.functional.gelu(gate, approximate="tanh") * up


def exact(case, seed):
    inp = _Inputs(case, seed)
    ytype = _TORCH[case.get("y", case["x"])]
    qmax = 127.0 if case["kind"] == "a8" else 7.0
    out = []
    for i, layer in enumerate(inp.layers):
        x = inp.x[i] if i < len(inp.x) else out[-1].to(ytype)  # the MLP's hidden units
        if inp.rot is not None:
            blk = case["rot"]
            v = x.double()[:, inp.perm.long()].view(x.shape[0], -1, blk)
            x = torch.einsum("mbi,bic->mbc", v, inp.rot.to(DEV)).reshape(x.shape).to(x.dtype)
        q, delta = _quantise(x, layer[3], inp.tables[i] if inp.tables else None, qmax)
        y = _product(q, delta, layer)
        out.append(_glue(y, layer[1], ytype) if layer[2] else y)
        if case["kind"] == "codes":
            u = q.to(torch.int16).bitwise_and(15).to(torch.uint8)
            return {"codes": u[:, 0::2] | (u[:, 1::2] << 4), "scale": delta[:, 0], "sum": q.sum(1).to(torch.int32),
                    "y": out[0]}
    return out


def tolerance(case):
    """Four times what the float32 path was measured to differ from `exact` by: the rounding of the output type (2.1e-4
    for f16, 1.7e-3 for bf16), and activation codes at a rounding tie that fall to the other side, each of which moves
    its whole row (3e-3 over a batch of 50 tokens with a step's scale, 3.9e-3 through the MLP's second quantiser; up to
    0.17 of a value).  Codes, sums and accumulators are whole numbers and stay the same."""
    y = case.get("y", case["x"])
    if case["kind"] == "mlp":
        return {"rel": 0.016, "max": 0.6}
    if y == "bf16":
        return {"rel": 0.008, "max": 0.25}
    return {"rel": 0.012 if case.get("step") else 0.0015, "max": 0.25}
