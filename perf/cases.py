"""What the framework's speed is measured on: the work its users have it do, through the C ABI
binding, over the range of models, batches and data types that it takes.

A case is one of these passes (``"pass"``):

``step``      ra_forward, ra_backward_truncated and ra_adapter_update on one batch: the
              fine-tuning step.  Loss, logits and gradients come back, and (``"params"``) the
              updated parameters.
``eval``      ra_forward alone, the held-out evaluation or a request served.  Loss and logits.
``pipelined`` two steps in the overlapped schedule: the frozen prefix of the second batch on a
              second stream while the first batch is in its suffix, backward and update.
``adapter``   ra_adapter_backward, the stand-alone fp32 adapter layer.

Values are those of a model in fine-tuning: N(0, 0.02) frozen weights but for the query and key
projections, which give attention scores of standard deviation 2 (so that a token attends to some
tokens and not to all alike), adapters whose up-projection has left zero (N(0, 5e-3)), hidden states
of unit variance, uniform labels, and a learning rate early in its warm-up.
"""
import math

import torch

from paper_2502_19864_gb300 import ringada as R

LR = 1e-6
ENC, SPAN, DEC = "cls", "span", "vocab"


def _model(name, kind, head, L, H, heads, F, m, B, S, depth, dtype="bf16", n_out=2, placement="houlsby", params=False):
    return {"name": name, "pass": kind, "head": head, "layers": L, "hidden": H, "heads": heads, "ffn": F, "m": m,
            "batch": B, "seq": S, "depth": depth, "dtype": dtype, "n_out": n_out, "placement": placement,
            "params": params}


def listed():
    return [
        # the smallest training step: a two-layer fp32 encoder of 128 tokens, one layer
        # unfrozen, where launches and latency are all there is
        _model("tiny_f32_step", "step", ENC, 2, 128, 2, 512, 16, 4, 32, 1, "f32", params=True),
        # an fp32 encoder at full depth, 385 ragged tokens, sizes that are no power of two
        _model("mid_f32_step", "step", ENC, 3, 192, 3, 768, 24, 5, 77, 3, "f32", params=True),
        # the stand-alone fp32 adapter backward at a BERT-base layer's size
        {"name": "adapter_f32_backward", "pass": "adapter", "tokens": 4096, "hidden": 768, "m": 64},
        # a small bf16 span encoder with ragged tiles in every kernel (300 tokens of 100)
        _model("small_bf16_step", "step", SPAN, 3, 256, 4, 1024, 32, 3, 100, 3, params=True),
        # one question of 128 tokens through a BERT-base-shaped model: the forward's latency
        _model("base_eval_b1", "eval", SPAN, 12, 768, 12, 3072, 64, 1, 128, 1),
        # BERT-base-shaped model, 32 x 128 tokens, early in the unfreezing schedule (d = 3)
        _model("base_step_d3", "step", ENC, 12, 768, 12, 3072, 64, 32, 128, 3),
        # question answering: two BERT-base blocks with the span head at its usual 384 tokens
        # and a bottleneck of 48 (adapters of 8 to 128 are all in use)
        _model("span_s384_m48_step", "step", SPAN, 2, 768, 12, 3072, 48, 12, 384, 2, params=True),
        # one BERT-large block that trains above one that does not need its input's gradient:
        # the block's forward and backward at 32 x 256 tokens
        _model("large_block_step", "step", ENC, 2, 1024, 16, 4096, 64, 32, 256, 2, params=True),
        # the same with the placement of one adapter after the feed-forward's add and norm
        _model("paper_block_step", "step", ENC, 2, 1024, 16, 4096, 64, 32, 256, 2, placement="post_ffn", params=True),
        # two batches of the overlapped schedule at half depth
        _model("base_pipelined_d6", "pipelined", ENC, 12, 768, 12, 3072, 64, 32, 128, 6, params=True),
        # two LLaMA-style decoder blocks and the 32000-word head on 8 x 1024 tokens
        _model("llama_block_step", "step", DEC, 2, 2048, 16, 5632, 128, 8, 1024, 2, n_out=32000, params=True),
        # the whole BERT-large-shaped step at half depth, the largest
        _model("large_step_d12", "step", ENC, 24, 1024, 16, 4096, 64, 32, 256, 12),
    ]


def _log(rng, lo, hi, to=1):
    """A multiple of ``to`` in [lo, hi], spread over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return int(min(hi, max(lo, round(v / to) * to)))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "eval", "pipelined", "adapter", "f32", "f32"])
    if kind == "adapter":
        return {"pass": "adapter", "tokens": _log(rng, 33, 8192), "hidden": _log(rng, 64, 2048, 4),
                "m": rng.choice([8, 16, 24, 32, 48, 64, 96, 128])}
    most = _flops(listed()[-1])
    while True:
        f32 = kind == "f32"
        dh = rng.choice([32, 64, 96, 128]) if f32 else rng.choice([64, 64, 128])
        heads = rng.choice([1, 2, 3, 4, 6]) if f32 else rng.choice([2, 3, 4, 6, 8, 12, 16])
        hidden = dh * heads
        if hidden % 64 or hidden > 2048 or hidden < 128:
            continue
        head = rng.choice([ENC, SPAN, DEC]) if kind not in ("pipelined",) else rng.choice([ENC, SPAN])
        tokens = _log(rng, 16, 512 if f32 else 8192)
        seq = min(tokens, _log(rng, 8, 200 if f32 else 1024))
        batch = max(1, min(256, tokens // seq))
        if head == DEC:
            n_out = 8 * _log(rng, 12, 400 if f32 else 4000)
            placement = "houlsby"
        else:
            n_out = 2 if head == SPAN else rng.choice([2, 2, 3, 5, 20])
            placement = rng.choice(["houlsby", "houlsby", "post_ffn"])
        layers = rng.choice([1, 2, 3]) if f32 else rng.choice([1, 2, 3, 4])
        depth = rng.randint(1, layers)
        if kind == "pipelined" and layers > 1:
            depth = rng.randint(1, layers - 1)
        c = {"pass": kind if not f32 else "step", "head": head, "layers": layers, "hidden": hidden, "heads": heads,
             "ffn": 64 * max(1, round(hidden * rng.choice([2, 2.75, 4]) / 64)),
             "m": rng.choice([8, 16, 24, 32, 48, 64, 96, 128]), "batch": batch, "seq": seq, "depth": depth,
             "dtype": "f32" if f32 else "bf16", "n_out": n_out, "placement": placement, "params": False}
        if _flops(c) <= most:
            return c


# ---- inputs -------------------------------------------------------------------------------

def _adapter_keys(c):
    return ["WdF", "WuF"] if c["placement"] == "post_ffn" else ["WdA", "WuA", "WdF", "WuF"]


def _shapes(c):
    H, F, m = c["hidden"], c["ffn"], c["m"]
    ad = {"WdA": (H, m), "WuA": (m, H), "WdF": (H, m), "WuF": (m, H)}
    if c["head"] == DEC:
        s = {"Wq": (H, H), "Wk": (H, H), "Wv": (H, H), "Wo": (H, H), "rms1_g": (H,), "Wg": (F, H), "Wu": (F, H),
             "Wd": (H, F), "rms2_g": (H,)}
        head = {"rmsf_g": (H,), "Wh": (c["n_out"], H)}
    else:
        s = {"Wqkv": (3 * H, H), "bqkv": (3 * H,), "Wo": (H, H), "bo": (H,), "ln1_g": (H,), "ln1_b": (H,),
             "W1": (F, H), "b1": (F,), "W2": (H, F), "b2": (H,), "ln2_g": (H,), "ln2_b": (H,)}
        head = {"Wh": (c["n_out"], H), "bh": (c["n_out"],)}
    s.update({k: ad[k] for k in _adapter_keys(c)})
    return s, head


def _inputs(c, seed):
    """Weights, and one or two batches, on the GPU: float32 tensors that hold values of the model's type."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    bf16 = c["dtype"] == "bf16"

    def value(shape, scale, mean=0.0):
        t = torch.randn(shape, generator=gen, device="cuda").mul_(scale).add_(mean)
        return t.to(torch.bfloat16).float() if bf16 else t

    def weight(key, shape):
        if key.endswith("_g"):
            return value(shape, 0.02, 1.0)
        if key in ("Wq", "Wk"):
            return value(shape, (2 / c["hidden"]) ** 0.5)
        if key == "Wqkv":
            return torch.cat([weight("Wq", (2 * shape[1], shape[1])), value((shape[1], shape[1]), 0.02)])
        return value(shape, 5e-3 if key in ("WuA", "WuF") else 0.02)

    layer, head = _shapes(c)
    layers = [{k: weight(k, s) for k, s in layer.items()} for _ in range(c["layers"])]
    top = {k: weight(k, s) for k, s in head.items()}
    batches = []
    for _ in range(2 if c["pass"] == "pipelined" else 1):
        x = value((c["batch"] * c["seq"], c["hidden"]), 1.0)
        shape, most = {ENC: ((c["batch"],), c["n_out"]), SPAN: ((c["batch"], 2), c["seq"]),
                       DEC: ((c["batch"], c["seq"]), c["n_out"])}[c["head"]]
        batches.append((x, torch.randint(0, most, shape, generator=gen, device="cuda", dtype=torch.int32)))
    return layers, top, batches


def _adapter_inputs(c, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    T, H, m = c["tokens"], c["hidden"], c["m"]
    n = lambda shape, scale=1.0: torch.randn(shape, generator=gen, device="cuda") * scale
    g, h, Wd, Wu = n((T, H), 1e-3), n((T, H)), n((H, m), 0.02), n((m, H), 5e-3)
    return g, h, (h.double() @ Wd.double()).float(), Wd, Wu


# ---- the passes ---------------------------------------------------------------------------

def _trained(c):
    """(layer, key) of every tensor that the pass trains.  The span head's bias has no
    gradient (a common shift leaves a softmax as it is), so it is not among them."""
    got = [(l, k) for l in range(c["layers"] - c["depth"], c["layers"]) for k in _adapter_keys(c)]
    return got + {ENC: [(-1, "Wh"), (-1, "bh")], SPAN: [(-1, "Wh")], DEC: []}[c["head"]]


def _named(c, of):
    """{name: of(layer, key)} of the trained tensors, a class head's weights and bias as one: the
    bias's gradient alone is a sum that nearly cancels."""
    got = {"%d.%s" % lk: of(*lk) for lk in _trained(c) if lk[0] >= 0}
    if c["head"] != DEC:
        got["head"] = of(-1, "Wh") if c["head"] == SPAN else of(-1, "Wh", "bh")
    return got


def prepare(case, seed):
    if case["pass"] == "adapter":
        T, H, m = case["tokens"], case["hidden"], case["m"]
        s = dict(zip(("g", "h", "z", "Wd", "Wu"), _adapter_inputs(case, seed)))
        empty = lambda *shape: torch.empty(shape, device="cuda")
        nb = R.ra_adapter_backward_scratch_bytes(T, H, m)
        s.update(case=case, dWd=empty(H, m), dWu=empty(m, H), dh=empty(T, H), nb=nb,
                 scratch=torch.empty(nb, dtype=torch.uint8, device="cuda"))
        return s
    c = case
    layers, top, batches = _inputs(c, seed)
    arch = {ENC: R.RA_ENCODER_POSTLN, SPAN: R.RA_ENCODER_POSTLN_SPAN, DEC: R.RA_DECODER_PRENORM}[c["head"]]
    cfg = R.make_cfg(arch, c["layers"], c["hidden"], c["heads"], c["ffn"], c["n_out"], c["batch"], c["seq"],
                     R.RA_BF16 if c["dtype"] == "bf16" else R.RA_F32, int(c["head"] != DEC), c["depth"],
                     1e-6 if c["head"] == DEC else 1e-12, 10000.0,
                     R.RA_ADAPTERS_POST_FFN if c["placement"] == "post_ffn" else R.RA_ADAPTERS_HOULSBY,
                     int(c["pass"] == "pipelined"))
    model = R.Model(cfg, c["m"], device="cuda:0")
    descs = [R.ra_tensor_desc(l, R.P[R.KEY_TO_PARAM[k]], t.data_ptr(), t.numel())
             for l, p in list(enumerate(layers)) + [(-1, top)] for k, t in p.items()]
    R.ra_set_weights(model.ctx, descs)
    R.ra_set_unfrozen_depth(model.ctx, c["depth"])
    layer = _shapes(c)[0]

    def view(get, l, *keys):
        at = [get(model.ctx, l, R.P[R.KEY_TO_PARAM[key]]) for key in keys]
        n = sum(a[1] for a in at)
        assert at[-1][0] + 4 * at[-1][1] == at[0][0] + 4 * n
        buf = model.buffers[1]
        off = at[0][0] - buf.data_ptr()
        return buf[off:off + 4 * n].view(torch.float32).view(layer[keys[0]] if l >= 0 else (n,))

    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    rows = c["batch"] if c["head"] == ENC else c["batch"] * c["seq"]
    s = dict(case=c, model=model, ctx=model.ctx, x=[x.to(dt) for x, _ in batches], labels=[y for _, y in batches],
             loss=[torch.zeros(1, device="cuda") for _ in batches],
             logits=[torch.zeros(rows, c["n_out"], device="cuda") for _ in batches])
    s["out"] = {"loss": s["loss"], "logits": s["logits"]}
    if c["pass"] != "eval":
        s["out"]["grads"] = _named(c, lambda l, *keys: view(R.ra_get_grad, l, *keys))
    if c["params"]:
        s["out"]["params"] = _named(c, lambda l, *keys: view(R.ra_get_param, l, *keys))
    if c["pass"] == "pipelined":
        s["streams"] = [torch.cuda.Stream(), torch.cuda.Stream()]
    return s


def run(state):
    s, c = state, state["case"]
    if c["pass"] == "adapter":
        p = {k: s[k].data_ptr() for k in ("g", "h", "z", "Wd", "Wu", "dWd", "dWu", "dh", "scratch")}
        R.ra_adapter_backward(p["g"], p["h"], p["z"], p["Wd"], p["Wu"], c["tokens"], c["hidden"], c["m"],
                              p["dWd"], p["dWu"], p["dh"], p["scratch"], s["nb"])
        return {"dWd": s["dWd"], "dWu": s["dWu"], "dh": s["dh"]}
    ctx, B, S, k = s["ctx"], c["batch"], c["seq"], c["layers"] - c["depth"]
    x, y, loss, logits = ([t.data_ptr() for t in s[n]] for n in ("x", "labels", "loss", "logits"))
    if c["pass"] != "pipelined":
        R.ra_forward(ctx, x[0], y[0], B, S, loss[0], logits[0])
        if c["pass"] == "step":
            R.ra_backward_truncated(ctx, k)
            R.ra_adapter_update(ctx, lr=LR)
        return s["out"]
    now = torch.cuda.current_stream()
    main, side = s["streams"]
    main.wait_stream(now)
    R.ra_forward_prefix(ctx, x[0], B, S, 0, main)
    side.wait_stream(main)
    R.ra_forward_prefix(ctx, x[1], B, S, 1, side)
    for i in (0, 1):
        R.ra_forward_suffix(ctx, i, y[i], loss[i], logits[i], main)
        R.ra_backward_truncated(ctx, k, main)
        R.ra_adapter_update(ctx, lr=LR, stream=main)
        main.wait_stream(side)
    now.wait_stream(main)
    return s["out"]


# ---- the work of a pass -------------------------------------------------------------------

def _flops(c):
    if c["pass"] == "adapter":
        return 10 * c["tokens"] * c["hidden"] * c["m"]
    L, H, F, m, S, T = c["layers"], c["hidden"], c["ffn"], c["m"], c["seq"], c["batch"] * c["seq"]
    dec = c["head"] == DEC
    dense = 2 * T * H * (4 * H + (3 if dec else 2) * F)
    attn = 4 * T * S * H * (0.5 if dec else 1)
    n_ad = len(_adapter_keys(c)) // 2
    adapter = 4 * T * H * m * n_ad
    head = 2 * c["n_out"] * H * (c["batch"] if c["head"] == ENC else T)
    f = L * (dense + attn + adapter) + head
    if c["pass"] != "eval":
        d = c["depth"]
        # layers above the lowest: every product's input gradient, attention twice and the
        # scores again; the lowest: with two adapters the feed-forward's, with one nothing
        f += (d - 1) * (dense + 2.5 * attn + 2.5 * adapter) + 2 * head
        f += 1.5 * adapter if n_ad == 1 else 2.25 * adapter + 2 * T * H * (3 if dec else 2) * F
    return int(f * (2 if c["pass"] == "pipelined" else 1))


def work(case):
    c = case
    if c["pass"] == "adapter":
        T, H, m = c["tokens"], c["hidden"], c["m"]
        return {"bytes": 4 * (3 * T * H + T * m + 4 * H * m), "flops": _flops(c)}
    es = 2 if c["dtype"] == "bf16" else 4
    layer, head = _shapes(c)
    rows = c["batch"] if c["head"] == ENC else c["batch"] * c["seq"]
    n = 2 if c["pass"] == "pipelined" else 1
    b = es * (c["layers"] * sum(math.prod(s) for s in layer.values()) + sum(math.prod(s) for s in head.values()))
    b += n * (es * c["batch"] * c["seq"] * c["hidden"] + 4 * rows * c["n_out"])
    if c["pass"] != "eval":
        trained = sum(math.prod((head if l < 0 else layer)[k]) for l, k in _trained(c))
        b += n * 4 * 7 * trained   # gradient out, master and two moments in and out
    return {"bytes": b, "flops": _flops(c)}


def tolerance(case):
    """About four times what the passes differ from 64 bits by, over the listed cases and some
    seventy drawn ones (worst: 6e-7 the stand-alone adapter, 3e-6 the fp32 models, 0.022 the
    bf16 models, where each layer's roundings travel through those after it)."""
    if case["pass"] == "adapter":
        return {"rel": 3e-6, "max": 3e-5}
    return {"rel": 1.2e-5, "max": 1e-4} if case["dtype"] == "f32" else {"rel": 0.03, "max": 0.6}


# ---- the same in 64 bits ------------------------------------------------------------------

def _norm(x, eps, g, b=None):
    if b is None:
        return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + eps) * g
    return torch.nn.functional.layer_norm(x, x.shape[-1:], g, b, eps)


def _adapter(a, p, branch):
    return a + torch.nn.functional.gelu(a @ p["Wd" + branch]) @ p["Wu" + branch]


def _attention(q, k, v, c):
    B, S, n = c["batch"], c["seq"], c["heads"]
    q, k, v = (t.view(B, S, n, -1).transpose(1, 2) for t in (q, k, v))
    if c["head"] == DEC:
        half = q.shape[-1] // 2
        at = torch.arange(S, device="cuda", dtype=torch.float64)[:, None] * (
            10000.0 ** (-torch.arange(half, device="cuda", dtype=torch.float64) / half))
        turn = lambda t: torch.cat([t[..., :half] * at.cos() - t[..., half:] * at.sin(),
                                    t[..., half:] * at.cos() + t[..., :half] * at.sin()], -1)
        q, k = turn(q), turn(k)
    s = q @ k.transpose(-1, -2) / math.sqrt(q.shape[-1])
    if c["head"] == DEC:
        s = s.masked_fill(torch.ones(S, S, dtype=torch.bool, device="cuda").triu(1), -math.inf)
    return (s.softmax(-1) @ v).transpose(1, 2).reshape(B * S, -1)


def _block(x, p, c):
    gelu, silu = torch.nn.functional.gelu, torch.nn.functional.silu
    if c["head"] == DEC:
        n = _norm(x, 1e-6, p["rms1_g"])
        a = _attention(n @ p["Wq"].T, n @ p["Wk"].T, n @ p["Wv"].T, c) @ p["Wo"].T
        x = x + _adapter(a, p, "A")
        n = _norm(x, 1e-6, p["rms2_g"])
        return x + _adapter((silu(n @ p["Wg"].T) * (n @ p["Wu"].T)) @ p["Wd"].T, p, "F")
    a = _attention(*(x @ p["Wqkv"].T + p["bqkv"]).chunk(3, -1), c) @ p["Wo"].T + p["bo"]
    two = c["placement"] == "houlsby"
    y = _norm(x + (_adapter(a, p, "A") if two else a), 1e-12, p["ln1_g"], p["ln1_b"])
    f = gelu(y @ p["W1"].T + p["b1"]) @ p["W2"].T + p["b2"]
    if two:
        return _norm(y + _adapter(f, p, "F"), 1e-12, p["ln2_g"], p["ln2_b"])
    return _adapter(_norm(y + f, 1e-12, p["ln2_g"], p["ln2_b"]), p, "F")


def _loss(x, top, labels, c):
    ce = torch.nn.functional.cross_entropy
    B, S, labels = c["batch"], c["seq"], labels.long()
    if c["head"] == DEC:
        z = _norm(x, 1e-6, top["rmsf_g"]) @ top["Wh"].T
        return ce(z, labels.view(-1)), z
    if c["head"] == SPAN:
        z = x @ top["Wh"].T + top["bh"]
        by = z.view(B, S, 2)
        return (ce(by[:, :, 0], labels[:, 0]) + ce(by[:, :, 1], labels[:, 1])) / 2, z
    z = x.view(B, S, -1)[:, 0] @ top["Wh"].T + top["bh"]
    return ce(z, labels), z


def exact(case, seed):
    if case["pass"] == "adapter":
        g, h, z, Wd, Wu = (t.double() for t in _adapter_inputs(case, seed))
        z.requires_grad_(True)
        s = torch.nn.functional.gelu(z)
        dz, = torch.autograd.grad(s, z, g @ Wu.T)
        return {"dWd": h.T @ dz, "dWu": s.detach().T @ g, "dh": g + dz @ Wd.T}
    c = case
    layers, top, batches = _inputs(c, seed)
    k = c["layers"] - c["depth"]
    find = lambda l, key: (top if l < 0 else layers[l])[key]
    at = _trained(c) if c["pass"] != "eval" else []
    state = {lk: find(*lk).double() for lk in at}
    losses, logits, grads = [], [], []
    m = {lk: torch.zeros_like(t) for lk, t in state.items()}
    v = {lk: torch.zeros_like(t) for lk, t in state.items()}
    for step, (x, labels) in enumerate(batches, 1):
        x = x.double()
        with torch.no_grad():
            for p in layers[:k]:
                x = _block(x, {n: t.double() for n, t in p.items()}, c)
        for t in state.values():
            t.requires_grad_(True)
        for l in range(k, c["layers"]):
            x = _block(x, {n: state.get((l, n), None) if (l, n) in state else t.double()
                           for n, t in layers[l].items()}, c)
        loss, z = _loss(x, {n: state[(-1, n)] if (-1, n) in state else t.double() for n, t in top.items()}, labels, c)
        losses.append(loss.detach().view(1))
        logits.append(z.detach())
        if not state:
            continue
        grads = dict(zip(state, torch.autograd.grad(loss, list(state.values()))))
        with torch.no_grad():
            for lk, g in grads.items():
                m[lk] = 0.9 * m[lk] + 0.1 * g
                v[lk] = 0.999 * v[lk] + 0.001 * g * g
                state[lk] = state[lk].detach() - LR * (m[lk] / (1 - 0.9 ** step)) / (
                    (v[lk] / (1 - 0.999 ** step)).sqrt() + 1e-8)
        del x, loss, z
    # the loss of a bf16 model is one rounded number: how far it falls from 64 bits is chance
    out = {"loss": losses if c["dtype"] == "f32" else None, "logits": logits}

    def whole(of):
        return _named(c, lambda l, *keys: of[l, keys[0]] if l >= 0 else torch.cat([of[l, k].flatten() for k in keys]))

    if state:
        out["grads"] = whole(grads)
    if c["params"]:
        out["params"] = whole(state)
    return out
