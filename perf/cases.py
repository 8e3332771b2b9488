"""The work whose speed is measured: calls a program that decodes with this library makes.

Most cases are single calls through the prepared calls of ``binding`` (what a loop over
layers and steps uses): one layer's state-masked attention, or one step's scoring and
transition; one is the 8B-shaped step (both), one the forward pass of the decoding driver's
model. ``listed`` names the workloads of ``workloads.py`` and their odd, ragged and typed
relatives; ``draw`` gives others of the same ranges. ``exact`` restates the computation in
64 bits (torch on the GPU), independently of the library.

A case's shape (sequence lengths, block positions, state counts) follows from the case
alone; the values, which positions hold which state, and the logits from the seed.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2608_26574_gb300 import binding as B
from paper_2608_26574_gb300 import decode

DEV = "cuda"
M, C, U = 0, 1, 2
TAU_C, TAU_U = 0.5, 0.8
LAMBDA, P0 = 0.5 ** (1.0 / 8.0), 0.1
THETA = 500000.0
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
_models: dict = {}


# ----------------------------------------------------------------------------- the cases

def _attn(name, dtype="bf16", hq=32, hkv=32, d=128, seqs=1, prompt_lo=512, prompt_hi=512, gen=256,
          block=32, index=-1, frac_m=0.5, frac_c=0.25, candidates=False, prefix=False, rope=0,
          image=0, shape_seed=0):
    """One attention call. index -1: each sequence at a block of its own; rope 0 none,
    1 interleaved pairs, 2 half pairs; image: leading rows with a spread of 1.5."""
    return dict(name=name, kind="attn", dtype=dtype, hq=hq, hkv=hkv, d=d, seqs=seqs,
                prompt_lo=prompt_lo, prompt_hi=prompt_hi, gen=gen, block=block, index=index,
                frac_m=frac_m, frac_c=frac_c, candidates=candidates, prefix=prefix, rope=rope,
                image=image, shape_seed=shape_seed)


def _score(name, dtype="bf16", seqs=1, block=32, vocab=126464, pad=0, frac_m=0.5, frac_c=0.25,
           extras=False):
    """One scoring call. pad: elements between the vocabulary and the row pitch; extras: the
    end-of-step outputs (next tokens, p_cur, entropy, margin, the next ordering key)."""
    return dict(name=name, kind="score", dtype=dtype, seqs=seqs, block=block, vocab=vocab, pad=pad,
                frac_m=frac_m, frac_c=frac_c, extras=extras)


def listed():
    step = _attn("step_8b", index=3)
    step.update(kind="step", vocab=126464)
    return [
        # the smallest call: one head group in fp32, a unit test's or a toy model's layer
        _attn("attn_tiny_f32", "f32", 4, 4, 64, prompt_lo=32, prompt_hi=32, gen=32, index=0,
              frac_m=0.4, frac_c=0.3),
        # fp32 inference of a small model over a ragged batch (validation runs, no bf16)
        _attn("attn_f32_batch", "f32", 8, 2, 128, seqs=4, prompt_lo=200, prompt_hi=700, gen=96,
              shape_seed=2),
        # a prefix-cached step of one 8B-class stream, q and k before RoPE: latency counts
        _attn("attn_8b_prefix_rope", index=5, prefix=True, rope=1),
        # the headline step of one stream: one 8B-class layer, then scoring of its block
        step,
        # one layer of a long-context grouped-query model
        _attn("attn_gqa", hq=28, hkv=4, prompt_lo=4096, prompt_hi=4096, gen=1024, block=64,
              index=8, frac_m=0.3, frac_c=0.4),
        # a serving batch of 32 requests of mixed lengths
        _attn("attn_ragged", seqs=32, prompt_lo=256, prompt_hi=2048, frac_m=0.5, shape_seed=4),
        # a multimodal batch (576 image rows each), RoPE in the call, half pairing
        _attn("attn_mm_rope", seqs=8, prompt_lo=704, prompt_hi=704, gen=512, index=10,
              frac_m=0.2, frac_c=0.6, rope=2, image=576),
        # head_dim 64, grouped heads, odd lengths, shadow rows for candidates only
        _attn("attn_d64_odd", hq=16, hkv=4, d=64, seqs=5, prompt_lo=333, prompt_hi=1501, gen=192,
              block=48, frac_m=0.3, frac_c=0.4, candidates=True, shape_seed=6),
        # the end of one stream's step with everything the next step needs
        _score("score_8b_extras", extras=True),
        # fp32 logits of a larger vocabulary, an odd vocabulary inside padded rows
        _score("score_f32_odd", "f32", 2, 64, 151643, pad=5, frac_m=0.3, frac_c=0.4),
        # the serving batch's scoring: 1024 rows
        _score("score_ragged", seqs=32),
        # a whole forward pass of the decoding driver's model over four prompts
        dict(name="model_forward", kind="model", layers=2, d_model=1024, heads=8, kv_heads=8,
             mlp=3072, vocab=32768, seqs=4, prompt=512, gen=128, block=32, index=1, frac_m=0.5,
             frac_c=0.25),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["attn", "attn", "attn", "attn", "f32", "score", "score", "model"])
    frac_m = round(rng.uniform(0.2, 0.8), 3)
    frac_c = round((1 - frac_m) * rng.uniform(0.3, 0.7), 3)
    if kind == "model":
        heads = rng.choice([4, 8])
        return dict(kind="model", layers=rng.randint(1, 3), d_model=128 * heads, heads=heads,
                    kv_heads=rng.choice([heads, heads // 4]), mlp=384 * heads,
                    vocab=8 * rng.randint(1024, 4096), seqs=rng.randint(1, 4),
                    prompt=_log(rng, 64, 1024), gen=rng.choice([64, 128, 256]), block=32,
                    index=rng.randint(0, 1), frac_m=frac_m, frac_c=frac_c)
    if kind == "score":
        c = _score("", rng.choice(["bf16", "bf16", "f32"]), _log(rng, 1, 32),
                   rng.choice([16, 32, 32, 64]), _log(rng, 1024, 152064), 0, frac_m, frac_c,
                   rng.random() < 0.5)
        while c["seqs"] * c["block"] > 1024:
            c["seqs"] //= 2
        c["pad"] = -c["vocab"] % 8
        del c["name"]
        return c
    f32 = kind == "f32"
    hq, hkv = rng.choice([(4, 4), (8, 2), (4, 1)] if f32 else
                         [(32, 32), (32, 8), (28, 4), (16, 16), (8, 2), (40, 8)])
    block = rng.choice([16, 32, 32, 48, 64, 128])
    c = _attn("", "f32" if f32 else "bf16", hq, hkv, rng.choice([64, 128, 128]),
              seqs=_log(rng, 1, 4 if f32 else 32), prompt_lo=_log(rng, 32, 500 if f32 else 3000),
              gen=block * rng.randint(1, 6), block=block, frac_m=frac_m, frac_c=frac_c,
              candidates=rng.random() < 0.3, prefix=rng.random() < 0.3,
              rope=rng.choice([0, 0, 1, 2]), shape_seed=rng.randrange(1 << 20))
    c["prompt_hi"] = int(c["prompt_lo"] * rng.uniform(1.0, 1.5))
    while work(c)["flops"] > (5e9 if f32 else 8e11) and c["seqs"] > 1:
        c["seqs"] -= 1
    del c["name"]
    return c


# ----------------------------------------------------------------------------- shapes

def _counts(c):
    """M, C and U positions of a block."""
    m = int(round(c["block"] * c["frac_m"]))
    n = min(int(round(c["block"] * c["frac_c"])), c["block"] - m)
    return m, n, c["block"] - m - n


def _shapes(c):
    """Per sequence: prompt, N, block start and shadow rows."""
    rng = random.Random(c["shape_seed"])
    out = []
    for _ in range(c["seqs"]):
        p = rng.randint(c["prompt_lo"], c["prompt_hi"])
        i = c["index"] if c["index"] >= 0 else rng.randrange(c["gen"] // c["block"])
        s = _counts(c)[1] if c["candidates"] else c["block"]
        out.append((p, p + c["gen"], p + i * c["block"], s))
    return out


def work(c):
    """The bytes and operations a pass cannot do without: every query, key, value and output
    row once, 4 d operations per (query row, position, head); a model also its weights once
    and its projections; scoring the shadow logits of every row and the original ones of M."""
    by = fl = 0
    if c["kind"] in ("attn", "step"):
        esz = 4 if c["dtype"] == "f32" else 2
        for p, n, _, s in _shapes(c):
            q = n + s - (p if c["prefix"] else 0)
            by += esz * c["d"] * (2 * q * c["hq"] + (3 if c["rope"] else 2) * (n + s) * c["hkv"])
            fl += 4 * c["d"] * q * n * c["hq"]
    if c["kind"] in ("score", "step"):
        m = _counts(c)[0] * c["seqs"]
        by += c["vocab"] * (4 if c["dtype"] == "f32" else 2) * (c["seqs"] * c["block"] + m)
    if c["kind"] == "model":
        n, b = c["prompt"] + c["gen"], c["block"]
        rows, hd = c["seqs"] * (n + b), 128
        per = c["d_model"] * (2 * c["heads"] * hd + 2 * c["kv_heads"] * hd + 3 * c["mlp"])
        fl = c["layers"] * (2 * rows * per + 4 * hd * rows * n * c["heads"])
        fl += 2 * 2 * c["seqs"] * b * c["d_model"] * c["vocab"]
        by = 2 * (c["layers"] * per + c["d_model"] * c["vocab"] + 2 * c["seqs"] * b * c["vocab"])
    return {"bytes": by, "flops": fl}


# ----------------------------------------------------------------------------- inputs

def _generators(seed):
    return torch.Generator().manual_seed(seed), torch.Generator(DEV).manual_seed(seed)


def _states(c, g):
    """States and last confidences of every block position, sequence by sequence."""
    nm, nc, nu = _counts(c)
    codes = torch.tensor([M] * nm + [C] * nc + [U] * nu, dtype=torch.uint8)
    st = torch.cat([codes[torch.randperm(c["block"], generator=g)] for _ in range(c["seqs"])])
    lo = torch.tensor([0.0, TAU_C, TAU_U])[st.long()]
    hi = torch.tensor([TAU_C, TAU_U, 1.0])[st.long()]
    return st, lo + (hi - lo) * (1 - torch.rand(len(st), generator=g))


def _sources(c, st):
    """Original positions of the shadow rows, sequence by sequence."""
    src = []
    for k, (_, _, b0, _) in enumerate(_shapes(c)):
        s = st[k * c["block"]:(k + 1) * c["block"]]
        at = torch.nonzero(s == C).flatten() if c["candidates"] else torch.arange(c["block"])
        src.append(at + b0)
    return src


def _attn_inputs(c, seed):
    g, gd = _generators(seed)
    sh = _shapes(c)
    rows = sum(n + s for _, n, _, s in sh)
    std = torch.full((rows, 1, 1), 1 / math.sqrt(c["d"]), device=DEV)
    if c["image"]:
        base = 0
        for _, n, _, s in sh:
            std[base:base + c["image"]] = 1.5
            base += n + s
    st, conf = _states(c, g)

    def t(h):
        x = torch.randn(rows, h, c["d"], generator=gd, device=DEV)
        return x.mul_(std).to(DTYPES[c["dtype"]])
    return t(c["hq"]), t(c["hkv"]), t(c["hkv"]), st, conf, _sources(c, st)


def _prepare_attn(c, seed):
    q, k, v, st, conf, src = _attn_inputs(c, seed)
    sh = np.array(_shapes(c), np.int32)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    call = B.AttentionCall(sh[:, 1], sh[:, 2], [c["block"]] * c["seqs"], sh[:, 3], st.to(DEV),
                           conf.to(DEV), torch.cat(src).to(torch.int32).to(DEV), status=status,
                           query_start=sh[:, 0] if c["prefix"] else None,
                           rope_theta=THETA if c["rope"] else 0.0,
                           rope_style=B.DARD_ROPE_HALF if c["rope"] == 2
                           else B.DARD_ROPE_INTERLEAVED)
    return dict(attn=call, q=q, k=k, v=v, o=torch.zeros_like(q),
                k_rope=torch.empty_like(k) if c["rope"] else None)


def _logits(c, g, gd):
    """Logits N(0, 3) with one planted entry per row that puts its confidence around the
    thresholds, in rows of vocab + pad entries (the padding is never read)."""
    rows, v = c["seqs"] * c["block"], c["vocab"]
    x = torch.randn(rows, v + c.get("pad", 0), generator=gd, device=DEV).mul_(3.0)
    top = math.log(v) + 4.5 + (8.6 * torch.rand(rows, generator=g) - 4.0)
    x[torch.arange(rows), torch.randint(v, (rows,), generator=g)] = top.to(DEV)
    return x.to(DTYPES[c["dtype"]])[:, :v]


def _score_inputs(c, seed):
    g, gd = _generators(seed + 1000003)
    st, _ = _states(c, g)
    lx, ls = _logits(c, g, gd), _logits(c, g, gd)
    return st, lx, ls, torch.randint(c["vocab"], (len(st),), generator=g, dtype=torch.int32)


def _prepare_score(c, seed, st=None):
    own, lx, ls, cur = _score_inputs(c, seed)
    st = (own if st is None else st).to(DEV)
    rows = len(st)

    def out(dtype):
        return torch.zeros(rows, dtype=dtype, device=DEV)
    o = dict(conf=out(torch.float32), token=out(torch.int32), state=out(torch.uint8),
             w=out(torch.float32), counts=torch.zeros(3 * c["seqs"], dtype=torch.int32, device=DEV))
    extra = {}
    if c.get("extras"):
        o.update(tokens=out(torch.int32), p_cur=out(torch.float32), entropy=out(torch.float32),
                 margin=out(torch.float32), order_key=out(torch.float32))
        extra = dict(cur_token=cur.to(DEV), mask_token=c["vocab"] - 1, order_mode=B.ORDER_ENTROPY,
                     **{k: o[k] for k in ("tokens", "p_cur", "entropy", "margin", "order_key")})
    ws = torch.zeros(B.dard_score_workspace_size(rows, c["vocab"], c["seqs"]), dtype=torch.uint8,
                     device=DEV)
    call = B.ScoreCall([c["block"]] * c["seqs"], st, TAU_C, TAU_U, LAMBDA, P0, o["conf"],
                       o["token"], o["state"], ws, w_out=o["w"], counts=o["counts"],
                       status=torch.zeros(1, dtype=torch.int32, device=DEV), **extra)
    return dict(score=call, lx=lx, ls=ls, out=o)


def _model(c):
    """The weights (seeded by themselves: a program loads one model and decodes many
    prompts with it)."""
    key = tuple(c[k] for k in ("layers", "d_model", "heads", "kv_heads", "mlp", "vocab"))
    if key not in _models:
        _models.clear()
        cfg = decode.ModelConfig(vocab=c["vocab"], d_model=c["d_model"], n_layers=c["layers"],
                                 hq=c["heads"], hkv=c["kv_heads"], head_dim=128, mlp=c["mlp"])
        _models[key] = decode.DLLM(cfg, device=DEV)
    return _models[key]


def _prepare_model(c, seed):
    model = _model(c)
    g, _ = _generators(seed)
    rng = np.random.default_rng(seed)
    prompts = [rng.integers(0, c["vocab"] - 1, c["prompt"]) for _ in range(c["seqs"])]
    gen = [rng.integers(0, c["vocab"] - 1, c["gen"]) for _ in range(c["seqs"])]
    b = decode.make_batch(prompts, c["gen"], c["block"], c["index"], gen, model.cfg, DEV)
    st, conf = _states(c, g)
    b.state, b.prev_conf = st.to(DEV), conf.to(DEV)
    return dict(model=model, batch=b)


def prepare(case, seed):
    if case["kind"] == "attn":
        return _prepare_attn(case, seed)
    if case["kind"] == "score":
        return _prepare_score(case, seed)
    if case["kind"] == "model":
        return _prepare_model(case, seed)
    s = _prepare_attn(case, seed)
    s.update(_prepare_score(case, seed, _states(case, _generators(seed)[0])[0]))
    return s


def run(s):
    if "model" in s:
        lx, ls = s["model"].forward(s["batch"])
        return {"logits_x": lx, "logits_s": ls}
    out = {}
    if "attn" in s:
        s["attn"](s["q"], s["k"], s["v"], s["o"], k_rope=s["k_rope"])
        out["o"] = s["o"]
        if s["k_rope"] is not None:
            out["k_rope"] = s["k_rope"]
    if "score" in s:
        s["score"](s["lx"], s["ls"])
        out.update(s["out"])
    return out


# ----------------------------------------------------------------------------- in 64 bits

def _rotate(x, pos, theta, style):
    """RoPE of [rows, heads, d] in 64 bits."""
    d = x.shape[-1]
    f = theta ** (-2.0 * torch.arange(d // 2, dtype=torch.float64, device=x.device) / d)
    a = pos.to(torch.float64)[:, None] * f
    co, si = a.cos()[:, None], a.sin()[:, None]
    p, q = (x[..., 0::2], x[..., 1::2]) if style == 1 else (x[..., :d // 2], x[..., d // 2:])
    r, t = p * co - q * si, p * si + q * co
    return torch.stack((r, t), -1).flatten(-2) if style == 1 else torch.cat((r, t), -1)


def _visible(n, b0, st, conf, src):
    """[rows, rows] bool: which key rows each query row attends (every position once, in the
    original or the shadow copy)."""
    nb, dev = len(st), st.device
    s = len(src)
    pos = torch.cat((torch.arange(n, device=dev), src))
    shadow = torch.arange(n + s, device=dev) >= n
    i = pos - b0
    inside = (i >= 0) & (i < nb)
    ic = i.clamp(0, nb - 1)
    si = torch.where(inside, st[ic].long(), torch.where(i < 0, U, M))
    ci = torch.where(inside, conf[ic], 0.0)
    own = shadow[:, None] & (i[:, None] == torch.arange(nb, device=dev))
    k = st.long()[None]
    si, sq = si[:, None], shadow[:, None]
    take_m = sq | (si != M)
    take_c = torch.where(si == M, sq, torch.where(si == U, torch.ones_like(sq),
                                                  ~(ci[:, None] <= conf[None]) | own))
    take = torch.where(k == U, own, torch.where(k == M, take_m, take_c))
    has = torch.zeros(nb, dtype=torch.bool, device=dev)
    has[src - b0] = True
    vis = torch.ones(n + s, n + s, dtype=torch.bool, device=dev)
    vis[:, b0:b0 + nb] = ~(take & has)
    vis[:, n:] = take[:, src - b0]
    return vis


def _attend(q, k, v, vis, q0):
    """Softmax attention in 64 bits of rows q0 on, [rows, heads, d]; zeros before."""
    o = torch.zeros_like(q)
    for h in range(q.shape[1]):
        g = h // (q.shape[1] // k.shape[1])
        z = (q[q0:, h] @ k[:, g].T) / math.sqrt(q.shape[-1])
        z.masked_fill_(~vis[q0:], -math.inf)
        o[q0:, h] = torch.softmax(z, -1) @ v[:, g]
    return o


def _exact_attn(c, seed):
    q, k, v, st, conf, src = _attn_inputs(c, seed)
    st, conf = st.to(DEV), conf.to(DEV)
    o = torch.zeros(q.shape, dtype=torch.float64, device=DEV)
    kr = torch.empty(k.shape, dtype=torch.float64, device=DEV) if c["rope"] else None
    base = 0
    for i, (p, n, b0, s) in enumerate(_shapes(c)):
        at, bl = slice(base, base + n + s), slice(i * c["block"], (i + 1) * c["block"])
        sq, sk, sv = q[at].double(), k[at].double(), v[at].double()
        sr = src[i].to(DEV)
        if c["rope"]:
            pos = torch.cat((torch.arange(n, device=DEV), sr))
            sq, sk = _rotate(sq, pos, THETA, c["rope"]), _rotate(sk, pos, THETA, c["rope"])
            kr[at] = sk
        vis = _visible(n, b0, st[bl], conf[bl], sr)
        o[at] = _attend(sq, sk, sv, vis, p if c["prefix"] else 0)
        base += n + s
    return {"o": o, "k_rope": kr} if c["rope"] else {"o": o}


def _exact_score(c, seed, st=None):
    own, lx, ls, cur = _score_inputs(c, seed)
    st = (own if st is None else st).to(DEV)
    rows, nb = len(st), c["block"]
    f64 = torch.float64
    conf, w = torch.zeros(rows, dtype=f64, device=DEV), torch.full((rows,), math.nan, dtype=f64,
                                                                   device=DEV)
    p_cur, ent, mar = (torch.zeros(rows, dtype=f64, device=DEV) for _ in range(3))

    def settle(r, z):
        lp = torch.log_softmax(z, 0)
        two = lp.topk(2).values.exp()
        conf[r], mar[r] = two[0], two[0] - two[1]
        ent[r] = -(lp.exp() * lp).sum()
        p_cur[r] = lp[int(cur[r])].exp()

    state = st.tolist()
    for r in range(rows):
        if state[r] != M:
            settle(r, ls[r].double())
    now = conf.tolist()
    for r in range(rows):
        if state[r] == M:
            b, p, d = r - r % nb, 0.0, 0.0
            for j in range(b, b + nb):
                if state[j] == C:
                    t = LAMBDA ** abs(r - j)
                    p, d = p + t * (now[j] > TAU_U), d + t * (now[j] <= TAU_C)
            w[r] = (p + P0) / (p + d + P0)
            settle(r, ls[r].double() + w[r] * (lx[r].double() - ls[r].double()))
    out = {"conf": conf, "token": None, "state": None, "w": w, "counts": None}
    if c.get("extras"):
        out.update(tokens=None, p_cur=p_cur, entropy=ent, margin=mar, order_key=-ent)
    return out


def _exact_model(c, seed):
    s = _prepare_model(c, seed)
    model, b = s["model"], s["batch"]
    h = model.emb.double()[b.tokens.long()]
    rows = len(h)

    def norm(x):
        return x * torch.rsqrt(x.pow(2).mean(-1, keepdim=True) + 1e-6)
    n, nb = c["prompt"] + c["gen"], c["block"]
    theta = model.cfg.rope_base
    for lay in model.layers:
        wt = {k: x.double() for k, x in lay.items()}
        a = norm(h)
        q = _rotate((a @ wt["wq"]).view(rows, c["heads"], 128), b.pos, theta, 1)
        k = _rotate((a @ wt["wk"]).view(rows, c["kv_heads"], 128), b.pos, theta, 1)
        v = (a @ wt["wv"]).view(rows, c["kv_heads"], 128)
        o = torch.empty_like(q)
        for i in range(c["seqs"]):
            at, bl = slice(i * (n + nb), (i + 1) * (n + nb)), slice(i * nb, (i + 1) * nb)
            b0 = int(b.block_start[i])
            vis = _visible(n, b0, b.state[bl], b.prev_conf[bl], b.shadow_src[bl].long())
            o[at] = _attend(q[at], k[at], v[at], vis, 0)
        h = h + o.flatten(1) @ wt["wo"]
        m = norm(h)
        h = h + (torch.nn.functional.silu(m @ wt["w1"]) * (m @ wt["w3"])) @ wt["w2"]
    h = norm(h)
    head = model.head.double()
    return {"logits_x": h[b.x_rows] @ head * model.cfg.logit_scale,
            "logits_s": h[b.s_rows] @ head * model.cfg.logit_scale}


def exact(case, seed):
    if case["kind"] == "attn":
        return _exact_attn(case, seed)
    if case["kind"] == "score":
        return _exact_score(case, seed)
    if case["kind"] == "model":
        return _exact_model(case, seed)
    out = _exact_attn(case, seed)
    out.update(_exact_score(case, seed, _states(case, _generators(seed)[0])[0]))
    return out
