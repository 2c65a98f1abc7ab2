"""The work that a user of this framework has it do: the BCMT token mixer as a
training step, a prefill, incremental decoding, and inside a whole model, each
through the public entry points (``layer.forward`` / ``layer.backward``,
``layer.Decoder``, ``gpt.GPT``).

``exact`` restates the mixer in plain float64 torch operations (Sec. 3.2-3.8 of
the paper; gradients by torch's autograd), without this repository's code.
"""

from __future__ import annotations

import math

import torch
import torch.nn.functional as F

from paper_2608_13578_gb300 import gpt, layer

DEV = "cuda"
DTYPES = {"bf16": torch.bfloat16, "fp32": torch.float32}
GRADS_X = ("dx", "dw_qkv", "dw_o", "dw_p", "dw_m", "dw_g")
GRADS_QKV = ("dq", "dk", "dv", "dw_o", "dw_p", "dw_m", "dw_g")


def _layer(name, B, T, D, H, L, dtype="bf16", backward=True, lo=0.8, hi=0.8, entry="x",
           honly=False, learn_decay=False):
    case = dict(kind="layer", B=B, T=T, D=D, H=H, L=L, dtype=dtype, backward=backward,
                decay_lo=lo, decay_hi=hi, entry=entry, honly=honly, learn_decay=learn_decay)
    return dict(name=name, **case) if name else case


def _decode(name, B, n, D, H, L, dtype="bf16"):
    case = dict(kind="decode", B=B, T=n, D=D, H=H, L=L, dtype=dtype, decay_lo=0.5, decay_hi=0.99)
    return dict(name=name, **case) if name else case


def _model(name, B, T, D, H, L, layers, mlp, vocab):
    case = dict(kind="model", B=B, T=T, D=D, H=H, L=L, layers=layers, mlp=mlp, vocab=vocab,
                dtype="bf16")
    return dict(name=name, **case) if name else case


def listed():
    return [
        # the smallest call: one short sequence through one layer in full precision
        # (the paper's recipe is plain fp32 PyTorch); latency and launches count
        _layer("fp32_forward_small", 1, 256, 128, 4, 32, "fp32", backward=False, lo=0.5, hi=0.99),
        # prefill: the forward of one prompt whose length is not a multiple of the block
        _layer("prefill_one_prompt", 1, 1500, 512, 8, 64, backward=False),
        # decoding one sequence over two blocks, token by token (interactive use)
        _decode("decode_one_sequence", 1, 128, 512, 8, 64),
        # decoding sixteen sequences in lockstep at a wider layer (serving)
        _decode("decode_sixteen", 16, 160, 1024, 16, 128),
        # a training step of one layer: the size the benchmark's headline is quoted on
        _layer("train_headline", 8, 1024, 512, 8, 64),
        # the same in fp32, for a user who trains or checks in full precision
        _layer("train_fp32", 8, 1024, 512, 8, 64, "fp32"),
        # the block-size sweep's largest block: attention over several key tiles
        _layer("train_block256", 16, 1024, 768, 12, 256),
        # the paper's own model shape (heads of 16) at the largest block of its table
        _layer("train_paper_l512", 16, 1024, 128, 8, 512),
        # the longest context of the sequence sweep: the largest case
        _layer("train_long_context", 4, 16384, 1024, 16, 128, lo=0.9, hi=0.999),
        # heads of 128, as wide models commonly have them
        _layer("train_wide_heads", 4, 2048, 1024, 8, 128),
        # odd sizes: a block of 48 tokens, heads of 96, a ragged last block, and a
        # learned per-channel decay
        _layer("train_odd_blocks", 4, 1000, 768, 8, 48, lo=0.5, hi=0.99, learn_decay=True),
        # a whole decoder's training pass (forward, loss, backward): the shape of the
        # decoder the benchmark trains, in 4 layers
        _model("model_pass", 8, 1024, 512, 8, 64, 4, 2048, 32000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _block(rng, hi=512):
    """Mostly the paper's powers of two, else any length."""
    if rng.random() < 0.6:
        return rng.choice([v for v in (16, 32, 64, 128, 256, 512) if v <= hi])
    return _log_int(rng, 16, hi)


def _width(rng, top=1024):
    """(D, H): head widths 16 to 128, the common ones most often."""
    while True:
        dh = rng.choice((16, 32, 64, 64, 64, 80, 96, 128, 128))
        D = rng.choice((64, 128, 192, 256, 384, 512, 640, 768, 1024))
        if D <= top and D % dh == 0:
            return D, D // dh


def draw(rng):
    u = rng.random()
    if u < 0.18:
        D, H = _width(rng)
        return _decode(None, _log_int(rng, 1, 24), rng.randint(96, 192), D, H, _block(rng, 256),
                       "fp32" if rng.random() < 0.15 else "bf16")
    if u < 0.24:
        D, H = rng.choice(((128, 8), (256, 4), (384, 6), (512, 8)))
        return _model(None, rng.randint(1, 8), rng.randint(128, 1024), D, H, _block(rng, 256),
                      rng.randint(1, 4), 4 * D, rng.choice((8192, 16000, 32000)))
    fp32 = rng.random() < 0.25
    D, H = _width(rng)
    L = _block(rng)
    most = 8192 if fp32 or D // H not in (16, 32, 64) or L not in (16, 32, 64, 128, 256, 512) \
        else 32768
    B = _log_int(rng, 1, 16)
    T = _log_int(rng, 64, min(16384, most // B))
    if rng.random() < 0.3:
        T = max(L, T // L * L)  # whole blocks
    T = min(T, most // B)
    lo = rng.choice((0.0, 0.5, 0.8, 0.9))
    hi = rng.choice((lo, 0.95, 0.999))
    return _layer(None, B, T, D, H, L, "fp32" if fp32 else "bf16", backward=rng.random() < 0.75,
                  lo=lo, hi=max(lo, hi), entry="qkv" if rng.random() < 0.15 else "x",
                  honly=rng.random() < 0.1, learn_decay=rng.random() < 0.2)


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _mixer_weights(case, g, dt):
    D = case["D"]
    std = D ** -0.5

    def normal(*shape):
        return (torch.randn(*shape, generator=g, device=DEV) * std).to(dt)

    t = dict(w_qkv=normal(D, 3 * D), w_o=normal(D, D), w_p=normal(D), w_m=normal(D, D),
             w_g=normal(D, D))
    lo, hi = case["decay_lo"], case["decay_hi"]
    t["decay"] = lo + (hi - lo) * torch.rand(D, generator=g, device=DEV)
    return t


def _layer_inputs(case, seed):
    g, dt = _gen(seed), DTYPES[case["dtype"]]
    shape = (case["B"], case["T"], case["D"])
    t = _mixer_weights(case, g, dt)
    if case["kind"] == "decode":
        shape = (case["T"], case["B"], case["D"])  # one contiguous row block per position
    names = ("q", "k", "v") if case.get("entry") == "qkv" else ("x",)
    for n in names + (("dy",) if case.get("backward") else ()):
        t[n] = torch.randn(*shape, generator=g, device=DEV).to(dt)
    return t


def _model_params(case, seed):
    """name -> value of every parameter, as the usual initialisations draw them."""
    g, D, m, V = _gen(seed), case["D"], case["mlp"], case["vocab"]
    out = {}

    def normal(name, *shape, std):
        out[name] = (torch.randn(*shape, generator=g, device=DEV) * std).bfloat16()

    def uniform(name, *shape, fan_in):
        u = torch.rand(*shape, generator=g, device=DEV) * 2 - 1
        out[name] = (u * fan_in ** -0.5).bfloat16()

    def norm(name):
        out[name + ".weight"] = torch.ones(D, device=DEV, dtype=torch.bfloat16)
        out[name + ".bias"] = torch.zeros(D, device=DEV, dtype=torch.bfloat16)

    normal("tok.weight", V, D, std=1.0)
    normal("pos", case["T"], D, std=0.02)
    for i in range(case["layers"]):
        p = "blocks.%d." % i
        norm(p + "ln1")
        for n, cols in (("w_qkv", 3 * D), ("w_o", D), ("w_m", D), ("w_g", D)):
            normal(p + "mix." + n, D, cols, std=D ** -0.5)
        normal(p + "mix.w_p", D, std=D ** -0.5)
        norm(p + "ln2")
        uniform(p + "fc1.weight", m, D, fan_in=D)
        uniform(p + "fc1.bias", m, fan_in=D)
        uniform(p + "fc2.weight", D, m, fan_in=m)
        uniform(p + "fc2.bias", D, fan_in=m)
    norm("ln_f")
    uniform("head.weight", V, D, fan_in=D)
    ids = torch.randint(V, (2, case["B"], case["T"]), generator=g, device=DEV)
    return out, ids[0], ids[1]


def prepare(case, seed):
    if case["kind"] == "model":
        values, ids, targets = _model_params(case, seed)
        c = gpt.GPTConfig(vocab=case["vocab"], D=case["D"], H=case["H"], layers=case["layers"],
                          mlp=case["mlp"], L=case["L"], T=case["T"])
        with torch.device(DEV):
            model = gpt.build(c)
        with torch.no_grad():
            for n, p in model.named_parameters():
                p.copy_(values[n])
        return dict(kind="model", model=model, ids=ids, targets=targets)
    t = _layer_inputs(case, seed)
    if case["kind"] == "decode":
        w = {n: t[n] for n in layer.WEIGHTS + ("decay",)}
        return dict(kind="decode", x=t["x"], dec=layer.Decoder(w, case["B"], case["H"], case["L"]))
    p = layer.params_for(case["B"], case["T"], case["D"], case["H"], case["L"], case["dtype"],
                         case["entry"] == "x", case["honly"])
    return dict(kind="layer", p=p, t=t, backward=case["backward"],
                learn_decay=case["learn_decay"])


# --------------------------------------------------------------------- run
def run(state):
    if state["kind"] == "layer":
        p, t = state["p"], state["t"]
        y, ws = layer.forward(p, t)
        if not state["backward"]:
            return {"y": y}
        return {"y": y, **layer.backward(p, t, ws, t["dy"], decay_grad=state["learn_decay"])}
    if state["kind"] == "decode":
        dec = state["dec"]
        dec.reset()
        return {"y": torch.stack([dec.step(x_t) for x_t in state["x"]])}
    model = state["model"]
    logits = model(state["ids"])
    loss = F.cross_entropy(logits.reshape(-1, logits.shape[-1]), state["targets"].reshape(-1))
    loss.backward()
    grads = {n: p.grad for n, p in model.named_parameters()}
    model.zero_grad(set_to_none=True)
    return {"logits": logits.detach(), "loss": loss.detach(), "grads": grads}


# -------------------------------------------------------------------- work
def work(case):
    B, T, D, L = case["B"], case["T"], case["D"], case["L"]
    es, n = (2 if case["dtype"] == "bf16" else 4), B * T
    mix = 8 * D * D + 2 * D * (min(L, T) + 1)  # W_qkv, W_o and causal attention, per token
    full = mix + 2 * D * D + 2 * D * D / L     # and the gate and the memory projection
    if case["kind"] == "decode":
        # the weights are needed at every position, with the block's keys and values
        weights = 6 * D * D * es + D * (es + 4)
        cache = B * (L + 1) * D * es
        return {"bytes": T * (weights + cache + 2 * B * D * es), "flops": n * full}
    if case["kind"] == "model":
        V, m, k = case["vocab"], case["mlp"], case["layers"]
        params = k * (6 * D * D + 5 * D + 2 * D * m + m + D) + (2 * V + T + 2) * D
        act = n * k * (4 * D + 2 * m) + 2 * n * V
        return {"bytes": 2 * (3 * params + 2 * act), "flops": 3 * n * (k * (full + 4 * D * m) + 2 * D * V)}
    x_in = case["entry"] == "x"
    flops = mix if case["honly"] else full
    if not x_in:
        flops -= 6 * D * D
    weights = (3 if x_in else 0) * D * D + D * D + (0 if case["honly"] else 2 * D * D + D)
    acts = (1 if x_in else 3) * n * D
    b = weights + acts + n * D
    if case["backward"]:
        b += weights + acts + n * D
    return {"bytes": b * es, "flops": (3 if case["backward"] else 1) * n * flops}


# ------------------------------------------------------------------- exact
def _mixer64(t, L, H, honly=False):
    """The mixer of Sec. 3.2-3.8 on float64 tensors (x or q, k, v and the weights)."""
    if "x" in t:
        q, k, v = (t["x"] @ t["w_qkv"]).chunk(3, dim=-1)
    else:
        q, k, v = t["q"], t["k"], t["v"]
    B, T, D = q.shape
    nb, dh = -(-T // L), D // H
    real = torch.arange(nb * L, device=DEV) < T  # the last block may be ragged

    def blocks(z):  # [B, nb, H, L, dh]
        z = F.pad(z, (0, 0, 0, nb * L - T))
        return z.view(B, nb, L, H, dh).transpose(2, 3)

    causal = torch.ones(L, L, dtype=torch.bool, device=DEV).triu(1)
    s = blocks(q) @ blocks(k).transpose(-1, -2) / math.sqrt(dh)
    a = torch.softmax(s.masked_fill(causal, -math.inf), -1)
    h = (a @ blocks(v)).transpose(2, 3).reshape(B, nb * L, D)[:, :T] @ t["w_o"]
    if honly:
        return h
    hb = F.pad(h, (0, 0, 0, nb * L - T)).view(B, nb, L, D)
    alpha = torch.softmax((hb @ t["w_p"]).masked_fill(~real.view(nb, L), -math.inf), -1)
    S = (alpha.unsqueeze(-1) * hb).sum(2)
    num, den, rows = torch.zeros_like(S[:, 0]), torch.zeros_like(t["decay"]), []
    for i in range(nb):
        num = t["decay"] * num + S[:, i]
        den = t["decay"] * den + 1
        rows.append(num / den)
    mem = F.pad(torch.stack(rows, 1) @ t["w_m"], (0, 0, 1, 0))[:, :nb]  # the one-block shift
    mem = mem.repeat_interleave(L, dim=1)[:, :T]
    return h + torch.sigmoid(h @ t["w_g"]) * mem


def _model64(p, ids, c):
    def norm(x, name):
        return F.layer_norm(x, (c["D"],), p[name + ".weight"], p[name + ".bias"])

    x = p["tok.weight"][ids] + p["pos"][: ids.shape[1]]
    for i in range(c["layers"]):
        b = "blocks.%d." % i
        t = {n: p[b + "mix." + n] for n in ("w_qkv", "w_o", "w_p", "w_m", "w_g")}
        t["decay"] = torch.full((c["D"],), 0.8, device=DEV).double()
        x = x + _mixer64(dict(t, x=norm(x, b + "ln1")), c["L"], c["H"])
        m = F.gelu(F.linear(norm(x, b + "ln2"), p[b + "fc1.weight"], p[b + "fc1.bias"]))
        x = x + F.linear(m, p[b + "fc2.weight"], p[b + "fc2.bias"])
    return F.linear(norm(x, "ln_f"), p["head.weight"])


def exact(case, seed):
    if case["kind"] == "model":
        values, ids, targets = _model_params(case, seed)
        p = {n: v.double().requires_grad_() for n, v in values.items()}
        logits = _model64(p, ids, case)
        loss = F.cross_entropy(logits.view(-1, case["vocab"]), targets.view(-1))
        loss.backward()
        return {"logits": logits.detach(), "loss": loss.detach(),
                "grads": {n: v.grad for n, v in p.items()}}
    t = {n: v.double() for n, v in _layer_inputs(case, seed).items()}
    if case["kind"] == "decode":
        t["x"] = t["x"].transpose(0, 1)
        return {"y": _mixer64(t, case["L"], case["H"]).transpose(0, 1).contiguous()}
    if not case["backward"]:
        return {"y": _mixer64(t, case["L"], case["H"], case["honly"])}
    names = GRADS_X if case["entry"] == "x" else GRADS_QKV
    names += ("d_decay",) if case["learn_decay"] else ()
    leaves = {}
    for n in names:
        leaves[n] = t[n[1:] if n != "d_decay" else "decay"].requires_grad_()
    y = _mixer64(t, case["L"], case["H"], case["honly"])
    grads = torch.autograd.grad(y, list(leaves.values()), t["dy"], allow_unused=True)
    out = {"y": y.detach()}
    for n, g in zip(leaves, grads):
        out[n] = torch.zeros_like(leaves[n]) if g is None else g
    return out
