"""The work that programs have this library do, as cases to be timed: sizes, inputs, one pass, what it cannot do without.

Four kinds of program:
  train    one training step of a quantized linear layer (Eq. 3-5): the weight quantizer, the forward product, both
           gradients.  With Q-EMA the weight is quantized once per step by the Q-EMA quantizer (and Q4 made from it), with
           the oscillation counters of Sec. 6.1 kept in the same pass or not; without it the forward pass quantizes the weight.
  mlp      one training step of fc1 -> GELU -> fc2 with the quantizations between the layers made in the products' epilogues.
  forward  evaluation: the forward pass alone, on a weight that was quantized when the model was loaded; any token count.
  weights  the optimizer's side of a step: Q-Ramping AdamW, the Q-EMA quantizer with its counters, Q4 for the next backward
           pass, and (every so many steps) the detection of oscillating weights.
"""
import math

import torch

import paper_2502_20853_b200 as mx

OUTLIER_CHANNELS, OUTLIER_GAIN = 4, 20.0     # activations: a few channels much larger than the rest
W_STD, DY_SCALE = 0.02, 1e-3
FLOOR, TRUNCATION_FREE = mx.SCALE_FLOOR, mx.SCALE_TRUNCATION_FREE
Q = 0.5 + 1.0 / 32.0                         # bytes of a quantized element: its code and its share of a scale


def _train(name, m, k, n, qema=False, osc=False, bias=False, floor=False, dw_bf16=False):
    return dict(name=name, kind="train", m=m, k=k, n=n, qema=qema, osc=osc, bias=bias, floor=floor, dw_bf16=dw_bf16)


def listed():
    return [
        # DeiT-Tiny fc1 on 1024 tokens: a small model or a small batch, where a step is a handful of short kernels
        _train("train_deit_tiny_fc1", 1024, 192, 768),
        # DeiT-Small at batch 128 x 197 tokens with Q-EMA, the method's own training recipe: an expanding layer ...
        _train("train_deit_small_fc1", 25216, 384, 1536, qema=True),
        # ... a contracting one with the oscillation counters, ...
        _train("train_deit_small_fc2", 25216, 1536, 384, qema=True, osc=True),
        # DeiT-Base qkv at batch 256 x 197 tokens
        _train("train_deit_base_qkv", 50432, 768, 2304, bias=True),
        # ViT-Large MLP at batch 256 x 197 tokens, the largest layers: short contraction and wide output, and the reverse
        _train("train_vit_large_fc1", 50432, 1024, 4096, bias=True),
        _train("train_vit_large_fc2", 50432, 4096, 1024, dw_bf16=True),
        # Swin-T: very many tokens with few channels (feature counts that fill no tile), ...
        _train("train_swin_stage1_fc1", 401408, 96, 384),
        # ... and the last stage, few tokens with many channels, with Microscaling's scale rule
        _train("train_swin_stage4_qkv", 6272, 768, 2304, floor=True),
        # DeiT-Small MLP, the two layers chained through the quantizing epilogues
        dict(name="mlp_deit_small", kind="mlp", m=25216, d=384, h=1536),
        # one image through DeiT-Small's fc1 (197 tokens): the smallest call
        dict(name="forward_one_image", kind="forward", m=197, k=384, n=1536, bias=True),
        # evaluation at batch 100 on DeiT-Base's qkv: a ragged token count
        dict(name="forward_eval_batch", kind="forward", m=19700, k=768, n=2304, bias=True),
        # the optimizer's side of a step on ViT-Large's fc1 weight
        dict(name="weights_vit_large_fc1", kind="weights", n=4096, k=1024, detect=True),
    ]


def _log(rng, lo, hi, step=1):
    """A multiple of `step` between lo and hi, spread over the logarithm."""
    return max(step, int(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step + 0.5) * step)


def draw(rng):
    kind = rng.choice(["train", "train", "train", "mlp", "forward", "weights"])
    while True:
        if kind == "forward":
            c = dict(kind=kind, m=_log(rng, 1, 50432), k=_log(rng, 96, 4096, 32), n=_log(rng, 96, 4096, 32), bias=rng.random() < 0.5)
            elems, flops = c["m"] * (c["k"] + c["n"]), c["m"] * c["k"] * c["n"]
        elif kind == "weights":
            c = dict(kind=kind, n=_log(rng, 96, 4096, 32), k=_log(rng, 96, 4096, 32), detect=rng.random() < 0.5)
            elems, flops = 0, 0
        elif kind == "mlp":
            d = _log(rng, 96, 1024, 32)
            c = dict(kind=kind, m=_log(rng, 512, 401408, 32), d=d, h=4 * d)
            elems, flops = c["m"] * 10 * d, c["m"] * 8 * d * d
        else:
            qema = rng.random() < 0.5
            c = _train("", _log(rng, 512, 401408, 32), _log(rng, 96, 4096, 32), _log(rng, 96, 4096, 32), qema=qema,
                       osc=qema and rng.random() < 0.5, bias=rng.random() < 0.5, floor=rng.random() < 0.25, dw_bf16=rng.random() < 0.25)
            del c["name"]
            elems, flops = c["m"] * (c["k"] + c["n"]), c["m"] * c["k"] * c["n"]
        if elems <= 50432 * 5120 and flops <= 50432 * 1024 * 4096:
            return c


# ---- inputs -----------------------------------------------------------------------------------------------------------
def _x(g, m, k):
    x = torch.randn((m, k), generator=g, device="cuda")
    x[:, torch.randperm(k, generator=g, device="cuda")[:OUTLIER_CHANNELS]] *= OUTLIER_GAIN
    return x.to(torch.bfloat16)


def _w(g, n, k):
    return (torch.randn((n, k), generator=g, device="cuda").clamp_(-2.0, 2.0) * W_STD).to(torch.bfloat16)


def _dy(g, m, n):
    """Heavy-tailed and small: Student-t with 3 degrees of freedom."""
    s = torch.zeros((m, n), device="cuda")
    for _ in range(3):
        s += torch.randn((m, n), generator=g, device="cuda").square_()
    return (torch.randn((m, n), generator=g, device="cuda") / (s / 3.0).sqrt_() * DY_SCALE).to(torch.bfloat16)


def _bias(g, n, wanted):
    return (torch.randn(n, generator=g, device="cuda") * 0.1).to(torch.bfloat16) if wanted else None


def _moved(g, w):
    """The weight some steps later (what the EMA and the previous step's buffers lag behind)."""
    return (w.float() + torch.randn(w.shape, generator=g, device="cuda") * (1e-3 * W_STD)).to(torch.bfloat16)


def _osc(g, w_prev, scale_mode=TRUNCATION_FREE):
    dist = [torch.rand(w_prev.shape, generator=g, device="cuda") * s for s in (1e-3, 2e-2)]
    return mx.OscState(w_prev.clone(), mx.quantize(w_prev, scale_mode=scale_mode), *dist)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s = dict(case=case, seed=0x5EED0000 + seed, status=mx.new_status())
    if case["kind"] == "train":
        m, k, n = case["m"], case["k"], case["n"]
        mode = FLOOR if case["floor"] else TRUNCATION_FREE
        s.update(mode=mode, x=_x(g, m, k), w=_w(g, n, k), dy=_dy(g, m, n), bias=_bias(g, n, case["bias"]),
                 dw_dtype=mx.OUT_BF16 if case["dw_bf16"] else mx.OUT_FP32,
                 ws=torch.empty(mx.linear_workspace_bytes(m, k, n), dtype=torch.uint8, device="cuda"))
        if case["qema"]:
            s.update(ema=s["w"].float(), wq=mx.QMat(n, k), wq_t=mx.QMat(k, n), osc=_osc(g, s["w"], mode) if case["osc"] else None)
            s["w"] = _moved(g, s["w"])
    elif case["kind"] == "mlp":
        m, d, h = case["m"], case["d"], case["h"]
        s.update(x=_x(g, m, d), w1=_w(g, h, d), w2=_w(g, d, h), dy=_dy(g, m, d),
                 # stands in for the derivative of the activation at Y1
                 slope=torch.rand((m, h), generator=g, device="cuda").to(torch.bfloat16),
                 ws=torch.empty(max(mx.linear_workspace_bytes(m, d, h), mx.linear_workspace_bytes(m, h, d)), dtype=torch.uint8, device="cuda"))
    elif case["kind"] == "forward":
        s.update(x=_x(g, case["m"], case["k"]), wq=mx.quantize(_w(g, case["n"], case["k"])), bias=_bias(g, case["n"], case["bias"]))
    else:
        n, k = case["n"], case["k"]
        w = _w(g, n, k)
        shape = (n, k)
        s.update(ema=w.float(), osc=_osc(g, w), wq=mx.QMat(n, k), wq_t=mx.QMat(k, n), w32=_moved(g, w).float(), w=_moved(g, w),
                 grad=torch.randn(shape, generator=g, device="cuda") * 1e-3, m=torch.randn(shape, generator=g, device="cuda") * 1e-3,
                 v=torch.rand(shape, generator=g, device="cuda") * 1e-6, acc=torch.zeros(shape, device="cuda"),
                 cnt=torch.zeros(shape, dtype=torch.uint8, device="cuda"),
                 # most weights are updated every step, the oscillating ones every sixth
                 n_w=1 + 5 * (torch.rand(shape, generator=g, device="cuda") < 0.1).to(torch.uint8))
    return s


# ---- one pass ---------------------------------------------------------------------------------------------------------
def _run_train(s):
    case, st, mode, seed = s["case"], s["status"], s["mode"], s["seed"]
    if case["qema"]:
        wq = mx.qema_quantize(s["w"], s["ema"], beta=0.998, scale_mode=mode, osc=s["osc"], out=s["wq"], dev_status=st)
        wq_t = mx.quantize_t(wq, scale_mode=mode, rounding=mx.ROUND_STOCHASTIC, seed=seed, stream_id=4, out=s["wq_t"], dev_status=st)
        ctx = mx.LinearCtx(mx.QMat(case["m"], case["k"]), wq, xq_t=mx.QMat(case["k"], case["m"]), seed=seed, wq_t=wq_t)
        y, ctx = mx.linear_fwd(s["x"], wq=wq, bias=s["bias"], scale_mode=mode, ctx=ctx, dev_status=st)
    else:
        y, ctx = mx.linear_fwd(s["x"], s["w"], bias=s["bias"], scale_mode=mode, bwd_seed=seed, dev_status=st)
    dx, dw = mx.linear_bwd(s["dy"], ctx, seed, scale_mode=mode, dw_dtype=s["dw_dtype"], workspace=s["ws"], dev_status=st)
    out = dict(y=y, dx=dx, dw=dw)
    if case["qema"]:
        out.update(ema=s["ema"], wq=ctx.wq.data)
        if s["osc"] is not None:
            out.update(dist_w=s["osc"].dist_w, dist_q=s["osc"].dist_q)
    return out


def _run_mlp(s):
    st, m, d, h = s["status"], s["case"]["m"], s["case"]["d"], s["case"]["h"]
    s1, s2 = s["seed"], s["seed"] + 10
    ctx1 = mx.LinearCtx(mx.QMat(m, d), mx.QMat(h, d), xq_t=mx.QMat(d, m), seed=s1, wq_t=mx.QMat(d, h))
    ctx2 = mx.LinearCtx(mx.QMat(m, h), mx.QMat(d, h), xq_t=mx.QMat(h, m), seed=s2, wq_t=mx.QMat(h, d))
    y1 = torch.empty((m, h), dtype=torch.bfloat16, device="cuda")
    dyq, dyq_t = mx.QMat(m, h), mx.QMat(h, m)
    up = mx.Epilogue(hook=mx.HOOK_GELU, y=y1, zq=ctx2.xq, zq_t=ctx2.xq_t, qp_t=(0, 1, s2, 6), chain=True)
    mx.linear_fwd(s["x"], s["w1"], ctx=ctx1, dev_status=st, epi=up)
    y2, _ = mx.linear_fwd(None, s["w2"], ctx=ctx2, dev_status=st)
    down = mx.Epilogue(hook=mx.HOOK_MULTIPLY, aux=s["slope"], zq=dyq, qp_row=(0, 1, s1, 3), zq_t=dyq_t, qp_t=(0, 1, s1, 5))
    _, dw2 = mx.linear_bwd(s["dy"], ctx2, s2, workspace=s["ws"], dev_status=st, epi_dx=down)
    dx, dw1 = mx.linear_bwd(None, ctx1, s1, workspace=s["ws"], dev_status=st, dyq=dyq, dyq_t=dyq_t)
    return dict(y1=y1, y2=y2, dx=dx, dw1=dw1, dw2=dw2)


def _run_weights(s):
    st, osc = s["status"], s["osc"]
    mx.qramp_adamw(s["w32"], s["grad"], s["m"], s["v"], s["acc"], s["cnt"], n_w=s["n_w"], step=100, w_bf16=s["w"])
    mx.qema_quantize(s["w"], s["ema"], beta=0.998, osc=osc, out=s["wq"], dev_status=st)
    mx.quantize_t(s["wq"], rounding=mx.ROUND_STOCHASTIC, seed=s["seed"], stream_id=4, out=s["wq_t"], dev_status=st)
    out = dict(w=s["w32"], w_bf16=s["w"], m=s["m"], v=s["v"], acc=s["acc"], cnt=s["cnt"], ema=s["ema"], wq=s["wq"].data,
               wq_t=s["wq_t"].data, dist_w=osc.dist_w, dist_q=osc.dist_q)
    if s["case"]["detect"]:
        out["n_w"], out["oscillating"] = mx.qramp_detect(osc.dist_w, osc.dist_q)
    return out


def run(state):
    kind = state["case"]["kind"]
    if kind == "train":
        return _run_train(state)
    if kind == "mlp":
        return _run_mlp(state)
    if kind == "forward":
        return mx.linear_fwd(state["x"], wq=state["wq"], bias=state["bias"], dev_status=state["status"])[0]
    return _run_weights(state)


# ---- what a pass cannot do without --------------------------------------------------------------------------------------
def work(case):
    """Inputs read once, outputs written once; operands that the step makes and uses itself (the quantized activations and
    gradients) are not counted.  The state a weight quantizer or the optimizer keeps is read and written."""
    kind = case["kind"]
    if kind == "weights":
        e = case["n"] * case["k"]
        adamw = 4 * 5 + 4 * 4 + 2 + 1 + 1 + 1          # w, m, v, acc, grad in; w, m, v, acc and the bf16 copy out; cnt both ways, n_w
        qema = 2 + 8 + 4 + 16 + 2 * Q + Q              # w, EMA, the previous weight, both distances, the previous codes; the codes
        return dict(bytes=e * (adamw + qema + Q + (1 if case["detect"] else 0)), flops=30 * e)
    if kind == "mlp":
        m, d, h = case["m"], case["d"], case["h"]
        return dict(bytes=2 * m * d * 4 + 2 * m * h * 2 + 2 * d * h * (2 + 4), flops=12 * m * d * h)
    m, k, n = case["m"], case["k"], case["n"]
    if kind == "forward":
        return dict(bytes=2 * m * (k + n) + Q * n * k, flops=2 * m * n * k)
    w = 2 + (2 if case["dw_bf16"] else 4) + ((8 + Q) if case["qema"] else 0) + ((4 + 16 + 2 * Q) if case["osc"] else 0)
    return dict(bytes=2 * m * (k + n) * 2 + w * k * n, flops=6 * m * n * k)


def tolerance(case):
    """The products accumulate in FP32 and are rounded to bf16: against products of the same operands in 64 bits they show
    1.7e-3 (2-norm) and 3.9e-3 (largest), which is the rounding alone.  The weights' state is FP32, element by element; its
    bf16 copy may round the other way."""
    return {"rel": 1e-5, "max": 0.008} if case["kind"] == "weights" else {"rel": 0.006, "max": 0.016}
