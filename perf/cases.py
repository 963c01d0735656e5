"""The work this library is measured on: the calls of a training step, at the
sizes of the repository's own workloads (C1..C6) and tests, each through the
public entry points with the buffers, workspaces and tables a training
program allocates once and keeps.

Kinds of case
  linear         one linear layer, forward and backward: the weight, the input
                 and the output gradient quantised (both copies), Fprop, then
                 Dgrad and Wgrad.  Blockwise or per-tensor scales, E4M3 or
                 E5M2 gradients, BF16 dW or an FP32 main-grad.
  norm_linear    RMSNorm fused into the quantiser, then the Fprop of a
                 projection (weights quantised once, as between two
                 optimizer steps).
  mlp_forward    the gated MLP: RMSNorm + quantise, gate/up Fprop, SwiGLU +
                 quantise, down Fprop.
  chain_backward a linear whose input gradient is the next linear's output
                 gradient: dY quantised, the Dgrad that quantises its own
                 output, the Wgrad added to the FP32 main-grad.
  weights        all weights of a model's layers quantised in one call, once
                 per optimizer step.
  muonh          the MuonH hyperball step over the weights of some layers.
  bf16_linear    the BF16 build of the three GEMMs.
"""
import math

import torch

import paper_2608_27370_gb300 as P
from paper_2608_27370_gb300 import workloads as W

DEV = "cuda"
EPS = 1e-6
ETA = 4.08e-4  # the paper's final Hyperball learning rate
MODELS = {"qwen2": W.QWEN2_1P5B_LINEARS, "qwen3": W.QWEN3_1P7B_LINEARS}
MAX_FLOPS = 6 * 32768 * 17920 * 1536  # the largest listed case


def listed():
    return [
        # C1: one per-tensor linear on 256 tokens -- the smallest training call, twelve launches of a few us
        dict(name="tensor_linear_m256", kind="linear", m=256, n=1536, k=1536, scaling="tensor", grad="e4m3", main=False),
        # the hybrid per-tensor recipe (E5M2 gradients) with no extent a multiple of the tiles
        dict(name="tensor_linear_ragged", kind="linear", m=4112, n=3968, k=1552, scaling="tensor", grad="e5m2", main=False),
        # a short blockwise linear with fewer output tiles than the GPU has SMs in every GEMM
        dict(name="block_linear_m640", kind="linear", m=640, n=1152, k=2560, scaling="block", grad="e4m3", main=False),
        # C6 o_proj: the paper's own model shape and micro-batch (2 x 4096 tokens), main-grad accumulation
        dict(name="block_linear_m8192", kind="linear", m=8192, n=2048, k=2048, scaling="block", grad="e4m3", main=True),
        # C5 gate_up: the largest linear of the 28-layer stack
        dict(name="block_linear_m32768", kind="linear", m=32768, n=17920, k=1536, scaling="block", grad="e4m3", main=False),
        # C5 attention input: RMSNorm and the qkv projection at 32768 tokens
        dict(name="norm_qkv_m32768", kind="norm_linear", m=32768, n=2048, k=1536),
        # the Qwen2-1.5B MLP on a short sequence
        dict(name="mlp_forward_m256", kind="mlp_forward", m=256, hidden=1536, ff=8960),
        # the Qwen3-1.7B MLP at the paper's micro-batch
        dict(name="mlp_forward_m8192", kind="mlp_forward", m=8192, hidden=2048, ff=6144),
        # C3 down projection, its input gradient handed on in FP8
        dict(name="chain_backward_m8192", kind="chain_backward", m=8192, n=1536, k=8960, grad="e4m3"),
        # once per optimizer step: the 112 weights of the paper's model
        dict(name="weights_28_layers", kind="weights", model="qwen3", layers=28),
        # once per optimizer step: a quarter of the Qwen2-1.5B stack's weights (one of four optimizer shards)
        dict(name="muonh_7_layers", kind="muonh", model="qwen2", layers=7),
        # C2 qkv in the BF16 build
        dict(name="bf16_linear_m8192", kind="bf16_linear", m=8192, n=2048, k=1536),
    ]


def _log(rng, lo, hi, step):
    """A multiple of step in [lo, hi], spread over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return int(min(hi, max(lo, step * round(v / step))))


def draw(rng):
    while True:
        c = _draw(rng)
        if work(c)["flops"] <= MAX_FLOPS:
            return c


def _draw(rng):
    kind = rng.choice(["linear", "linear", "linear", "norm_linear", "mlp_forward", "mlp_forward", "chain_backward",
                       "weights", "muonh", "bf16_linear"])
    _, n, k = rng.choice(MODELS[rng.choice(["qwen2", "qwen3"])])
    own = rng.random() < 0.5  # a model's linear, or any sizes
    if kind in ("weights", "muonh"):
        return dict(kind=kind, model=rng.choice(["qwen2", "qwen3"]), layers=_log(rng, 1, 28 if kind == "weights" else 7, 1))
    if kind == "bf16_linear":
        m = _log(rng, 128, 16384, 8)
        return dict(kind=kind, m=m, n=n if own else _log(rng, 128, 8192, 8), k=k if own else _log(rng, 128, 8192, 8))
    if kind == "linear" and rng.random() < 0.4:
        return dict(kind=kind, m=_log(rng, 128, 16384, 16), n=n if own else _log(rng, 128, 8192, 16),
                    k=k if own else _log(rng, 128, 8192, 16), scaling="tensor", grad=rng.choice(["e4m3", "e5m2"]),
                    main=rng.random() < 0.3)
    m = _log(rng, 128, 32768, 128)
    if not own:
        n, k = _log(rng, 256, 17920, 128), _log(rng, 256, 8960, 128)
    if kind == "linear":
        return dict(kind=kind, m=m, n=n, k=k, scaling="block", grad=rng.choice(["e4m3", "e4m3", "e5m2"]),
                    main=rng.random() < 0.3)
    if kind == "norm_linear":
        return dict(kind=kind, m=m, n=n, k=k)
    if kind == "mlp_forward":
        hidden, ff = rng.choice([(1536, 8960), (2048, 6144), (_log(rng, 256, 4096, 128), _log(rng, 512, 8960, 128))])
        return dict(kind=kind, m=m, hidden=hidden, ff=ff)
    return dict(kind=kind, m=m, n=n, k=k, grad=rng.choice(["e4m3", "e5m2"]))


# ------------------------------------------------------------------ inputs
def _fmt(name):
    return P.E5M2 if name == "e5m2" else P.E4M3


def _act(m, k, seed):
    """Rows as a projection receives them: RMSNorm of heavy-tailed rows."""
    return W.rmsnorm_rows_f32(W.student_t3_f32((m, k), DEV, seed)).to(torch.bfloat16)


def _pre_norm(m, k, seed):
    """Residual-stream rows ahead of the norm, and the norm's gain."""
    h = W.student_t3_f32((m, k), DEV, seed)
    h *= torch.exp2(W.normal_f32((m, 1), 2.0, DEV, seed + 1))
    gamma = (1.0 + W.normal_f32((k,), 0.1, DEV, seed + 2)).to(torch.bfloat16)
    return h.to(torch.bfloat16), gamma


def _operands(rows, cols, scaling, role, fmt):
    """Empty quantised copies of a [rows, cols] tensor, as a program keeps them."""
    mk = lambda r, c: P.FP8Operand(torch.empty((r, c), dtype=torch.uint8, device=DEV),  # noqa: E731
                                   P.empty_scales(r, c, scaling, role, DEV), fmt, scaling, role)
    amax = torch.zeros(1, dtype=torch.int32, device=DEV) if scaling == P.SCALE_TENSOR else None
    return P.Quantized(mk(rows, cols), mk(cols, rows), amax)


def _empty(*shape, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device=DEV)


def _workspace(*gemms):
    return _empty(max([16] + [P.puro_fp8_workspace_size(*g) for g in gemms]), dtype=torch.uint8)


def _weight(n, k, seed):
    """A weight and its quantised copies, made once (it changes once per optimizer step)."""
    w = W.normal_bf16((n, k), 0.02, DEV, seed)
    return w, P.quantize(w, P.E4M3, P.SCALE_BLOCK, P.ROLE_WEIGHT)


def prepare(case, seed):
    c, kind, seed = dict(case), case["kind"], seed * 1000 + 17
    if kind == "linear":
        m, n, k = c["m"], c["n"], c["k"]
        sc = P.SCALE_BLOCK if c["scaling"] == "block" else P.SCALE_TENSOR
        c.update(sc=sc, x=_act(m, k, seed), w=W.normal_bf16((n, k), 0.02, DEV, seed + 10),
                 dy=W.normal_bf16((m, n), 1e-3, DEV, seed + 20), xq=_operands(m, k, sc, P.ROLE_ACT, P.E4M3),
                 wq=_operands(n, k, sc, P.ROLE_WEIGHT, P.E4M3), dyq=_operands(m, n, sc, P.ROLE_ACT, _fmt(c["grad"])),
                 y=_empty(m, n), dx=_empty(m, k), ws=_workspace((m, n, k), (m, k, n), (n, k, m)))
        c["dw"] = W.normal_f32((n, k), 1e-2, DEV, seed + 30) if c["main"] else _empty(n, k)
        if sc == P.SCALE_BLOCK:
            c["table"] = P.weight_table([(c["w"], c["wq"])])
    elif kind == "norm_linear":
        m, n, k = c["m"], c["n"], c["k"]
        c["h"], c["gamma"] = _pre_norm(m, k, seed)
        c["w"], c["wq"] = _weight(n, k, seed + 10)
        c.update(rstd=_empty(m, dtype=torch.float32), xq=_operands(m, k, P.SCALE_BLOCK, P.ROLE_ACT, P.E4M3),
                 y=_empty(m, n), ws=_workspace((m, n, k)))
    elif kind == "mlp_forward":
        m, hid, ff = c["m"], c["hidden"], c["ff"]
        c["h"], c["gamma"] = _pre_norm(m, hid, seed)
        c["w1"], c["w1q"] = _weight(2 * ff, hid, seed + 10)
        c["w2"], c["w2q"] = _weight(hid, ff, seed + 20)
        c.update(rstd=_empty(m, dtype=torch.float32), xq=_operands(m, hid, P.SCALE_BLOCK, P.ROLE_ACT, P.E4M3),
                 aq=_operands(m, ff, P.SCALE_BLOCK, P.ROLE_ACT, P.E4M3), gu=_empty(m, 2 * ff), y=_empty(m, hid),
                 ws=_workspace((m, 2 * ff, hid), (m, hid, ff)))
    elif kind == "chain_backward":
        m, n, k = c["m"], c["n"], c["k"]
        c["w"], c["wq"] = _weight(n, k, seed + 10)
        c["x"] = _act(m, k, seed)
        c.update(dy=W.normal_bf16((m, n), 1e-3, DEV, seed + 20), xq=P.quantize(c["x"]),
                 dyq=_operands(m, n, P.SCALE_BLOCK, P.ROLE_ACT, _fmt(c["grad"])),
                 dxq=_operands(m, k, P.SCALE_BLOCK, P.ROLE_ACT, _fmt(c["grad"])), dx=_empty(m, k),
                 main=W.normal_f32((n, k), 1e-2, DEV, seed + 30), ws=_workspace((n, k, m)))
    elif kind == "weights":
        shapes = [(n, k) for _ in range(c["layers"]) for _, n, k in MODELS[c["model"]]]
        total = sum(n * k for n, k in shapes)
        flat = W.normal_bf16((total,), 0.02, DEV, seed)
        # one buffer for all codes and one for all scales: each weight's copies are views of them
        codes = _empty(2 * total, dtype=torch.uint8)
        scales = _empty(sum(P.puro_fp8_scale_bytes(n, k) + P.puro_fp8_scale_bytes(k, n) for n, k in shapes), dtype=torch.uint8)
        entries, at, at_q, at_s = [], 0, 0, 0
        for n, k in shapes:
            ops = []
            for r, red in ((n, k), (k, n)):
                sb = P.puro_fp8_scale_bytes(r, red)
                ops.append(P.FP8Operand(codes[at_q:at_q + n * k].view(r, red), scales[at_s:at_s + sb].view(P.scale_vec_shape(r, red)),
                                        P.E4M3, P.SCALE_BLOCK, P.ROLE_WEIGHT))
                at_q, at_s = at_q + n * k, at_s + sb
            entries.append((flat[at:at + n * k].view(n, k), P.Quantized(ops[0], ops[1])))
            at += n * k
        c.update(flat=flat, codes=codes, scales=scales, entries=entries, table=P.weight_table(entries))
    elif kind == "muonh":
        sizes = [n * k for _ in range(c["layers"]) for _, n, k in MODELS[c["model"]]]
        w = W.normal_f32((sum(sizes),), 0.02, DEV, seed)
        u = W.normal_f32((sum(sizes),), 1.0, DEV, seed + 10)
        wb = _empty(sum(sizes))
        mats, at = [], 0
        for n in sizes:
            s = slice(at, at + n)
            mats.append((w[s], u[s], wb[s], 0.02 * math.sqrt(n)))
            at += n
        c.update(w=w, u=u, wb=wb, mats=mats, sums=_empty(len(sizes), 3, dtype=torch.float64),
                 ws=_empty(max(16, P.puro_muonh_grouped_workspace_size(mats)), dtype=torch.uint8))
    else:
        m, n, k = c["m"], c["n"], c["k"]
        x, w, dy = _act(m, k, seed), W.normal_bf16((n, k), 0.02, DEV, seed + 10), W.normal_bf16((m, n), 1e-3, DEV, seed + 20)
        c.update(x=x, w=w, dy=dy, w_t=w.t().contiguous(), x_t=x.t().contiguous(), dy_t=dy.t().contiguous(),
                 y=_empty(m, n), dx=_empty(m, k), dw=_empty(n, k))
    c["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    return c


# --------------------------------------------------------------- one pass
def run(s):
    return globals()["_run_" + s["kind"]](s)


def _run_linear(s):
    st, sc, x, dy = s["status"], s["sc"], s["xq"], s["dyq"]
    if sc == P.SCALE_BLOCK:
        P.puro_fp8_quantize_weights(s["table"], P.E4M3, dev_status=st)
    else:
        P.quantize(s["w"], P.E4M3, sc, P.ROLE_WEIGHT, out=s["wq"], dev_status=st)
    P.quantize(s["x"], P.E4M3, sc, P.ROLE_ACT, out=x, dev_status=st)
    P.puro_fp8_linear_fprop(x.rowwise, s["wq"].rowwise, s["y"], s["ws"], dev_status=st)
    P.quantize(s["dy"], dy.rowwise.fmt, sc, P.ROLE_ACT, out=dy, dev_status=st)
    if s["main"]:
        P.puro_fp8_linear_dgrad(dy.rowwise, s["wq"].colwise, s["dx"], s["ws"], dev_status=st)
        P.puro_fp8_linear_wgrad_main_grad(dy.colwise, x.colwise, s["dw"], s["ws"], dev_status=st)
    else:
        P.puro_fp8_linear_backward(dy.rowwise, s["wq"].colwise, s["dx"], dy.colwise, x.colwise, s["dw"], s["ws"],
                                   dev_status=st)
    return {"y": s["y"], "dx": s["dx"], "dw": s["dw"], "xq": _bytes(x), "wq": _bytes(s["wq"]), "dyq": _bytes(dy)}


def _run_norm_linear(s):
    x = s["xq"]
    P.puro_fp8_quantize_rmsnorm(s["h"], s["gamma"], EPS, P.E4M3, s["rstd"], None, x.rowwise.data, x.rowwise.scale,
                                x.colwise.data, x.colwise.scale, dev_status=s["status"])
    P.puro_fp8_linear_fprop(x.rowwise, s["wq"].rowwise, s["y"], s["ws"], dev_status=s["status"])
    return {"rstd": s["rstd"], "y": s["y"], "xq": _bytes(x)}


def _run_mlp_forward(s):
    st, x, a, ff = s["status"], s["xq"], s["aq"], s["ff"]
    P.puro_fp8_quantize_rmsnorm(s["h"], s["gamma"], EPS, P.E4M3, s["rstd"], None, x.rowwise.data, x.rowwise.scale,
                                x.colwise.data, x.colwise.scale, dev_status=st)
    P.puro_fp8_linear_fprop(x.rowwise, s["w1q"].rowwise, s["gu"], s["ws"], dev_status=st)
    P.puro_fp8_quantize_swiglu(s["gu"][:, :ff], s["gu"][:, ff:], P.E4M3, None, a.rowwise.data, a.rowwise.scale,
                               a.colwise.data, a.colwise.scale, dev_status=st)
    P.puro_fp8_linear_fprop(a.rowwise, s["w2q"].rowwise, s["y"], s["ws"], dev_status=st)
    return {"rstd": s["rstd"], "gu": s["gu"], "y": s["y"], "xq": _bytes(x), "aq": _bytes(a)}


def _run_chain_backward(s):
    st, dy, dx = s["status"], s["dyq"], s["dxq"]
    P.quantize(s["dy"], dy.rowwise.fmt, P.SCALE_BLOCK, P.ROLE_ACT, out=dy, dev_status=st)
    P.puro_fp8_linear_dgrad_quantize(dy.rowwise, s["wq"].colwise, dx.rowwise.fmt, s["dx"], dx.rowwise.data,
                                     dx.rowwise.scale, dx.colwise.data, dx.colwise.scale, dev_status=st)
    P.puro_fp8_linear_wgrad_main_grad(dy.colwise, s["xq"].colwise, s["main"], s["ws"], dev_status=st)
    return {"dx": s["dx"], "main": s["main"], "dyq": _bytes(dy), "dxq": _bytes(dx)}


def _run_weights(s):
    P.puro_fp8_quantize_weights(s["table"], P.E4M3, dev_status=s["status"])
    return {"codes": s["codes"], "scales": s["scales"]}


def _run_muonh(s):
    P.puro_muonh_step_grouped(s["mats"], ETA, s["sums"], s["ws"])
    return {"w": s["w"], "wb": s["wb"], "sums": s["sums"]}


def _run_bf16_linear(s):
    m, n, k, st = s["m"], s["n"], s["k"], s["status"]
    P.puro_bf16_linear_fprop(s["x"], s["w"], s["y"], m, n, k, dev_status=st)
    P.puro_bf16_linear_dgrad(s["dy"], s["w_t"], s["dx"], m, n, k, dev_status=st)
    P.puro_bf16_linear_wgrad(s["dy_t"], s["x_t"], s["dw"], m, n, k, dev_status=st)
    return {"y": s["y"], "dx": s["dx"], "dw": s["dw"]}


def _bytes(q):
    """Codes and scales of both copies."""
    return [q.rowwise.data, q.rowwise.scale, q.colwise.data, q.colwise.scale]


# --------------------------------------------------- work and tolerances
def _copies(rows, cols, block=True):
    """Bytes of the two FP8 copies of a [rows, cols] tensor and their scales."""
    return 2 * rows * cols + (4 * rows * -(-cols // 512) + 4 * cols * -(-rows // 512) if block else 8)


def work(case):
    kind = case["kind"]
    if kind in ("weights", "muonh"):
        shapes = [(n, k) for _ in range(case["layers"]) for _, n, k in MODELS[case["model"]]]
        total = sum(n * k for n, k in shapes)
        if kind == "muonh":  # W and u in, W and its BF16 copy out
            return {"bytes": 14 * total, "flops": 10 * total}
        return {"bytes": 2 * total + sum(_copies(n, k) for n, k in shapes), "flops": 2 * total}
    m = case["m"]
    if kind == "mlp_forward":
        h, f = case["hidden"], case["ff"]
        b = 2 * m * h + 3 * h * f + 4 * m + _copies(m, h) + 2 * m * 2 * f + _copies(m, f) + 2 * m * h
        return {"bytes": b, "flops": 6 * m * h * f}
    n, k = case["n"], case["k"]
    if kind == "norm_linear":
        return {"bytes": 2 * m * k + n * k + 4 * m + _copies(m, k) + 2 * m * n, "flops": 2 * m * n * k}
    if kind == "bf16_linear":  # each operand in both orientations, three outputs
        return {"bytes": 6 * (m * n + m * k + n * k), "flops": 6 * m * n * k}
    if kind == "chain_backward":  # dY, the weight's and the input's transposed copies, main-grad in and out
        b = 2 * m * n + 2 * n * k + m * k + 8 * n * k + _copies(m, n) + 2 * m * k + _copies(m, k)
        return {"bytes": b, "flops": 4 * m * n * k}
    block = case["scaling"] == "block"
    b = 4 * (m * n + m * k) + (2 + (8 if case["main"] else 2)) * n * k
    b += _copies(m, n, block) + _copies(m, k, block) + _copies(n, k, block)
    return {"bytes": b, "flops": 6 * m * n * k}


def tolerance(case):
    kind = case["kind"]
    if kind == "weights":
        return "exact"
    if kind == "muonh":
        # fp32 sums of up to 64 values a thread, three fp32 roundings an element; a BF16 copy may round the
        # other way (2^-8 of the value) where the fp32 value lies at a boundary
        return {"rel": 1e-4, "max": 8e-3}
    # BF16 outputs are 1.7e-3 off the 64-bit result (rel), and one rounding the other way is 2^-8 of a value; the
    # codes of given inputs are exact.  Codes of computed values (normalised rows, silu(gate) * up, dX) follow
    # BF16 values that lie at a rounding boundary: up to 5e-5 of them differ from the 64-bit computation's.
    if kind in ("mlp_forward", "norm_linear", "chain_backward"):
        return {"rel": 7e-3, "max": 0.03, "differ": 2e-4}
    return {"rel": 7e-3, "max": 0.016}


# ------------------------------------------------------ the same in 64 bits
_TORCH8 = {"e4m3": (torch.float8_e4m3fn, 448.0), "e5m2": (torch.float8_e5m2, 57344.0)}


def _pow2_at_least(ratio):
    """The smallest power of two not below each ratio (1 for 0), no smaller than 2^-127."""
    m, e = torch.frexp(ratio)
    p = torch.where(m > 0.5, e, e - 1).clamp(min=-127)
    return torch.where(ratio > 0, torch.ldexp(torch.ones_like(ratio), p), torch.ones_like(ratio))


def _fake_rows(x, fmt="e4m3"):
    """x rounded to FP8 with a power-of-two scale per 1x128 group of a row, as fp64."""
    dt, top = _TORCH8[fmt]
    v = x.double().view(x.shape[0], -1, 128)
    s = _pow2_at_least(v.abs().amax(-1, keepdim=True) / top)
    return ((v / s).float().to(dt).double() * s).view(x.shape)


def _fake_blocks(w):
    n, k = w.shape
    v = w.double().view(n // 128, 128, k // 128, 128)
    s = _pow2_at_least(v.abs().amax((1, 3), keepdim=True) / 448.0)
    return ((v / s).float().to(torch.float8_e4m3fn).double() * s).view(n, k)


def _fake_tensor(x, fmt="e4m3"):
    """One scale a tensor: codes of fp32(x * scale), times fp32(1 / scale)."""
    dt, top = _TORCH8[fmt]
    scale = torch.tensor(top, device=x.device) / x.abs().amax().float()
    return (x.float() * scale).clamp(-top, top).to(dt).double() * (1.0 / scale).double()


def _rmsnorm(h, gamma):
    rstd = 1.0 / (h.double().square().mean(-1) + EPS).sqrt()
    return rstd, (h.double() * rstd[:, None] * gamma.double()).to(torch.bfloat16)


def exact(case, seed):
    s, kind = prepare(case, seed), case["kind"]
    if kind == "weights":
        return None
    none4 = [None] * 4
    if kind == "muonh":
        ws, at, sums = torch.empty_like(s["w"], dtype=torch.float64), 0, []
        for w, u, _, r in s["mats"]:
            w, u = w.double(), u.double()
            sums.append(torch.stack([(w * w).sum(), (w * u).sum(), (u * u).sum()]))
            t = w - ETA * r * u / u.norm()
            ws[at:at + w.numel()] = r * t / t.norm()
            at += w.numel()
        return {"w": ws, "wb": ws, "sums": torch.stack(sums)}
    if kind == "bf16_linear":
        x, w, dy = s["x"].double(), s["w"].double(), s["dy"].double()
        return {"y": x @ w.t(), "dx": dy @ w, "dw": dy.t() @ x}
    if kind == "norm_linear":
        rstd, x = _rmsnorm(s["h"], s["gamma"])
        return {"rstd": rstd, "y": _fake_rows(x) @ _fake_blocks(s["w"]).t(), "xq": none4}
    if kind == "mlp_forward":
        rstd, x = _rmsnorm(s["h"], s["gamma"])
        gu = _fake_rows(x) @ _fake_blocks(s["w1"]).t()
        g, u = gu.to(torch.bfloat16).double().chunk(2, 1)
        a = (torch.nn.functional.silu(g) * u).to(torch.bfloat16)
        del g, u
        return {"rstd": rstd, "gu": gu, "y": _fake_rows(a) @ _fake_blocks(s["w2"]).t(), "xq": none4, "aq": none4}
    t = lambda v, fmt="e4m3": _fake_rows(v.t().contiguous(), fmt)  # noqa: E731  (groups along the tokens)
    if kind == "chain_backward":
        dx = _fake_rows(s["dy"], s["grad"]) @ _fake_blocks(s["w"])
        main = s["main"].double() + t(s["dy"], s["grad"]) @ t(s["x"]).t()
        return {"dx": dx, "main": main, "dyq": none4, "dxq": none4}
    grad, start = s["grad"], s["dw"].double() if s["main"] else 0.0
    if s["scaling"] == "block":
        w = _fake_blocks(s["w"])
        y = _fake_rows(s["x"]) @ w.t()
        dx = _fake_rows(s["dy"], grad) @ w
        dw = t(s["dy"], grad) @ t(s["x"]).t()
        none = [none4] * 3
    else:
        x, w, dy = _fake_tensor(s["x"]), _fake_tensor(s["w"]), _fake_tensor(s["dy"], grad)
        y, dx, dw = x @ w.t(), dy @ w, dy.t() @ x
        # the two scale outputs of a copy are fp32 numbers of their own
        si = [(1.0 / (torch.tensor(f, device=DEV) / v.abs().amax().float())).double().reshape(1)
              for v, f in ((s["x"], 448.0), (s["w"], 448.0), (s["dy"], _TORCH8[grad][1]))]
        none = [[None, v, None, v] for v in si]
    return {"y": y, "dx": dx, "dw": start + dw, "xq": none[0], "wq": none[1], "dyq": none[2]}
