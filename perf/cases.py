"""What a user of this library has it do, as a list of measured cases.

Every case goes through the public entry points (``PardEngine``,
``cod_select`` and the C ABI's allocation-free acceptance) on seeded random
models of the repository's own shapes.  Model cases build the engine, its
weights and (where the pass needs one) the prompt's KV cache in ``prepare``,
as a serving program has them in hand; ``run`` is one pass.

First tokens and sampled tokens are drawn at a temperature so high (1e8) that
the random numbers alone decide them wherever later outputs depend on them:
on random-init weights the top two of 128256 logits are often closer than two
correct implementations' roundings, and one flipped token would change every
logit after it.  The temperature changes no work.  Passes whose tokens are a
plain argmax or a draw at T = 1 return the logits that decide them.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import synthetic as S
from paper_2504_18583_gb300 import pard

T_FLAT = 1e8  # logits / T vanish beside the Gumbel noise: the noise's largest entry wins, the lowest index on ties
PAGE = 16

MODELS = {
    # target shape, draft shape
    "tiny": (S.WORKLOADS["tiny"].target, S.WORKLOADS["tiny"].draft),
    "8b": (S.TARGET_8B, S.DRAFT_1B),
    "70b": (S.TARGET_70B, S.DRAFT_1B),
}
# the batch-16 configuration's prompt lengths, uniform in [128, 2048]
LENS16 = "1922,1532,161,1596,1020,1843,1698,1705,940,247,232,657,267,785,660,691"


def listed():
    def model(name, kind, which, layers, dlayers, lens, K, **kw):
        return dict(name=name, kind=kind, model=which, layers=layers, dlayers=dlayers, lens=lens, K=K,
                    sample=kw.get("sample", False), steps=kw.get("steps", 0))

    return [
        # training-data construction: the kept rows of one 2048-token sample's mask subtasks
        dict(name="cod_2048_k8", kind="cod", n=2048, K=8, r=0.5, r_min=0.05),
        # acceptance inside an engine that plans its own memory: one greedy sequence (smallest call),
        # and a batch of 16 sampled ones (reads all logits of both models)
        dict(name="accept_greedy_b1_k8", kind="accept", batch=1, K=8, vocab=128256, sample=False),
        dict(name="accept_sample_b16_k6", kind="accept", batch=16, K=6, vocab=128256, sample=True),
        # the smallest model pass: the 4-layer check configuration, all launch latency
        model("verify_tiny_b1", "verify", "tiny", 4, 2, "32", 4),
        # batch-1 decoding of the 8B / 1B pair, the headline configuration: its two passes
        model("draft_1b_b1_ctx512", "draft", "8b", 1, 16, "512", 8),
        model("verify_8b_b1_ctx512", "verify", "8b", 32, 1, "512", 8),
        # batch 16 with ragged contexts: sampled draft (its logits are kept) and verify
        model("draft_1b_b16_ragged", "draft", "8b", 1, 16, LENS16, 6, sample=True),
        model("verify_8b_b16_ragged", "verify", "8b", 8, 1, LENS16, 6),
        # 70B widths at the 4096-token context (a slice of the depth: three engines fit the card)
        model("verify_70b_b1_ctx4096", "verify", "70b", 4, 1, "4096", 8),
        # prompt pass: one 512-token prompt at full depth, and a batch of short ragged ones
        model("prefill_8b_512", "prefill", "8b", 32, 16, "512", 4),
        model("prefill_8b_b4_ragged", "prefill", "8b", 8, 4, "37,301,120,64", 4),
        # a whole short request: prompt pass and four sampled decode steps
        model("generate_8b_64", "generate", "8b", 32, 16, "64", 8, sample=True, steps=4),
    ]


def draw(rng):
    def log_int(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    kind = rng.choice(["cod", "accept", "draft", "draft", "verify", "verify", "verify", "prefill", "generate"])
    if kind == "cod":
        return dict(kind="cod", n=log_int(16, 2048), K=rng.randint(2, 8), r=round(rng.uniform(0.3, 0.9), 3),
                    r_min=rng.choice([0.0, 0.05, 0.1]))
    if kind == "accept":
        return dict(kind="accept", batch=log_int(1, 16), K=rng.randint(1, 6), vocab=8 * log_int(256, 16032),
                    sample=rng.random() < 0.5)
    which = rng.choice(["tiny", "8b", "8b", "8b", "70b"])
    K = rng.randint(2, 8)
    sample = rng.random() < 0.5
    steps = 0
    if kind in ("draft", "verify"):
        batch = log_int(1, 24)
        top = min(2048, 16384 // batch)
        if which == "70b":
            batch, top = log_int(1, 8), 512
        lens = [log_int(16, top) for _ in range(batch)]
        layers, dlayers = (rng.randint(2, 4), 1) if kind == "verify" else (1, rng.randint(2, 6))
        if kind == "verify":
            sample = False
            if rng.random() < 0.2:
                K = 0  # autoregressive decoding: one row per sequence
    elif kind == "prefill":
        batch = log_int(1, 6)
        lens = [log_int(8, 1500 // batch) for _ in range(batch)]
        layers, dlayers = rng.randint(2, 6 if which != "70b" else 2), rng.randint(1, 4)
    else:
        batch = log_int(1, 8)
        lens = [log_int(8, 128) for _ in range(batch)]
        layers, dlayers, steps, sample = rng.randint(2, 4), rng.randint(1, 4), rng.randint(1, 4), True
    return dict(kind=kind, model=which, layers=layers, dlayers=dlayers, lens=",".join(str(x) for x in lens), K=K,
                sample=sample, steps=steps)


# ---- inputs ------------------------------------------------------------------
def _lens(case):
    return [int(x) for x in case["lens"].split(",")]


def _shapes(case):
    t, d = MODELS[case["model"]]
    return t.replace(n_layers=case["layers"]), d.replace(n_layers=case["dlayers"])


def _weights(shape, seed):
    """N(0, 0.02) matrices, norm gains around 1, bf16, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)

    def mat(name):
        dims = shape.tensor_shape(name)
        if name.endswith("norm"):
            return (1.0 + 0.1 * torch.randn(dims, generator=g, device="cuda")).to(torch.bfloat16)
        return torch.empty(dims, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=g)

    w = {n: mat(n) for n in S.GLOBAL_TENSORS}
    w["layers"] = [{n: mat(n) for n in S.LAYER_TENSORS} for _ in range(shape.n_layers)]
    return w


def _prompts(case, seed, vocab):
    g = torch.Generator().manual_seed(seed * 7 + 1)
    return [torch.randint(0, vocab - 1, (L,), generator=g).tolist() for L in _lens(case)]


def _candidates(case, seed, vocab):
    g = torch.Generator().manual_seed(seed * 7 + 2)
    return torch.randint(0, vocab - 1, (len(_lens(case)), max(case["K"], 1)), generator=g)


def _n_new(case):
    return 1 + max(case["steps"], 4) * (case["K"] + 1)


def _accept_inputs(case, seed):
    """Target and draft logits that agree as a draft trained for the target does, and the draft's candidates."""
    B, K, V = case["batch"], case["K"], case["vocab"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    y = 2.0 * torch.randn((B, K + 1, V), generator=g, device="cuda")
    z = y[:, :K] + 0.5 * torch.randn((B, K, V), generator=g, device="cuda")
    if case["sample"]:
        u = torch.rand(z.shape, generator=g, device="cuda").clamp_(1e-7, 1 - 1e-6)
        d = (z - torch.log(-torch.log(u))).argmax(-1)
    else:
        d = y[:, :K].argmax(-1)
        hit = torch.rand((B, K), generator=g, device="cuda") < 0.8
        d = torch.where(hit, d, (d + 1) % V)
    return y, z, d.to(torch.int32).contiguous()


def prepare(case, seed):
    s = dict(case=case, seed=seed)
    if case["kind"] == "cod":
        return s
    if case["kind"] == "accept":
        s["y"], s["z"], s["d"] = _accept_inputs(case, seed)
        s["len"] = torch.empty(case["batch"], dtype=torch.int32, device="cuda")
        s["emitted"] = torch.empty((case["batch"], case["K"] + 1), dtype=torch.int32, device="cuda")
        return s
    t, d = _shapes(case)
    lens, K, n_new = _lens(case), case["K"], _n_new(case)
    s["prompts"] = _prompts(case, seed, t.vocab)
    s["cand"] = _candidates(case, seed, t.vocab).to("cuda", torch.int32)
    max_ctx = max(lens) + n_new + 2 * K + 16
    n_pages = sum(-(-(L + n_new + 2 * K) // PAGE) for L in lens)
    g = torch.Generator().manual_seed(seed * 7 + 3)
    s["eng"] = eng = pard.PardEngine(t, _weights(t, 2 * seed), d, _weights(d, 2 * seed + 1), max_batch=len(lens),
                                     max_k=max(K, 1), max_ctx=max_ctx, n_pages=n_pages,
                                     page_order_target=torch.randperm(n_pages, generator=g).tolist(),
                                     page_order_draft=torch.randperm(n_pages, generator=g).tolist())
    if case["kind"] in ("draft", "verify"):
        eng.prefill(s["prompts"], n_new, K, True, T_FLAT, seed)
    else:
        eng.batch, eng.K = len(lens), K  # the outputs' sizes; run() prefills
    s["out"] = [eng.alloc_step_outputs(want_logits=True) for _ in range(max(case["steps"], 1))]
    return s


# ---- one pass ----------------------------------------------------------------
def run(s):
    case, seed = s["case"], s["seed"]
    kind = case["kind"]
    if kind == "cod":
        keep, counts = pard.cod_select(case["n"], case["K"], case["r"], case["r_min"], seed, 3)
        return {"keep": keep, "counts": counts}
    if kind == "accept":
        code = pard.lib().pard_accept_noalloc(
            s["y"].data_ptr(), s["z"].data_ptr() if case["sample"] else None, s["d"].data_ptr(), case["batch"],
            case["K"], case["vocab"], int(case["sample"]), 1.0, seed, 5, s["len"].data_ptr(), s["emitted"].data_ptr(),
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert code == 0, pard.pard_last_error()
        return {"accept_len": s["len"], "emitted": s["emitted"]}
    eng, out = s["eng"], s["out"]
    if kind == "draft":
        eng.draft(out[0], case["sample"], 1.0, seed, 1)
        return {"draft_logits": out[0]["draft_logits"]}
    if kind == "verify":
        eng.verify(out[0], s["cand"] if case["K"] else None, 1.0)
        return {"logits": out[0]["logits"]}
    first = eng.prefill(s["prompts"], _n_new(case), case["K"], True, T_FLAT, seed)
    if kind == "prefill":
        eng.verify(out[0], s["cand"], 1.0)
        return {"first": first, "logits": out[0]["logits"]}
    for i, o in enumerate(out):
        eng.step(o, True, T_FLAT, seed, i + 1)
    return {"first": first, "emitted": [o["emitted"] for o in out], "accept_len": [o["accept_len"] for o in out],
            "kv_slots": [o["kv_slots"] for o in out], "logits": out[-1]["logits"]}


# ---- what a pass cannot do without ---------------------------------------------
def _pass_work(shape, rows, ctx, head_rows, read_ctx):
    """One forward: `rows` and `ctx` (positions before them) per sequence; head_rows logits rows."""
    n = sum(rows)
    mats = sum(int(np.prod(shape.tensor_shape(k))) for k in S.LAYER_TENSORS)
    head = int(np.prod(shape.tensor_shape("lm_head")))
    pairs = sum(r * c + r * (r + 1) // 2 for r, c in zip(rows, ctx))
    flops = 2 * shape.n_layers * mats * n + 2 * head * head_rows
    flops += 4 * shape.n_layers * shape.n_q_heads * shape.head_dim * pairs
    kv = shape.kv_bytes_per_token()
    by = 2 * (shape.n_layers * mats + (head if head_rows else 0)) + 2 * shape.d_model * n + kv * n
    by += kv * sum(ctx) if read_ctx else 0
    return by, flops


def work(case):
    if case["kind"] == "cod":
        rows = (case["K"] - 1) * case["n"]
        return {"bytes": 4 * (rows + case["K"]), "flops": 40 * rows}
    if case["kind"] == "accept":
        B, K, V = case["batch"], case["K"], case["vocab"]
        rows = B * (K + 1) + (B * K if case["sample"] else 0)
        return {"bytes": 4 * rows * V + 4 * B * (2 * K + 2), "flops": 4 * rows * V}
    t, d = _shapes(case)
    lens, K, B = _lens(case), case["K"], len(_lens(case))
    by = fl = 0

    def add(w, logit_rows=0):
        nonlocal by, fl
        by, fl = by + w[0] + 4 * logit_rows * t.vocab, fl + w[1]

    if case["kind"] in ("prefill", "generate"):
        zero = [0] * B
        add(_pass_work(t, lens, zero, B, False))
        add(_pass_work(d, lens, zero, 0, False))
    if case["kind"] == "draft":
        add(_pass_work(d, [K] * B, lens, B * K, True), B * K)
    if case["kind"] in ("verify", "prefill"):
        add(_pass_work(t, [K + 1] * B, lens, B * (K + 1), True), B * (K + 1))
    for i in range(case["steps"]):
        ctx = [n + i * (K + 1) for n in lens]
        add(_pass_work(d, [K if i == 0 else 2 * K] * B, ctx, B * K, True), B * K)
        add(_pass_work(t, [K + 1] * B, ctx, B * (K + 1), True), B * (K + 1))
    return {"bytes": by, "flops": fl}


def tolerance(case):
    if case["kind"] in ("cod", "accept"):
        return "exact"
    # Measured against exact(): the error grows with the square root of the depth (0.9e-3 at 2 and 3.7e-3 at 32
    # layers of the 8B widths, 0.9e-3 at 16 of the 1B, 2.5e-3 at 4 of the 70B, 0.3e-3 at 4 of the tiny ones), and the
    # largest difference is six to eight times it: about four times those.
    t, d = _shapes(case)
    shape = d if case["kind"] == "draft" else t
    unit = 6e-4 if shape.d_model <= 256 else 1e-3 if shape.d_model <= 2048 else 2.5e-3 if shape.d_model <= 4096 else 5e-3
    rel = unit * math.sqrt(max(shape.n_layers, 2))
    return {"rel": rel, "max": 8 * rel}


# ---- the same values in 64 bits --------------------------------------------------
def _philox_argmax(seed, stream, step, b, i, vocab):
    """The token of the largest Gumbel noise (a draw from the uniform distribution)."""
    M = np.uint64(0xFFFFFFFF)
    v = np.arange((vocab + 3) // 4, dtype=np.uint64)
    c = [v, np.full_like(v, (stream << 16) | i), np.full_like(v, b), np.full_like(v, step)]
    k = [seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF]
    for r in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k[0]), p1 & M, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k[1]), p0 & M]
        k = [(k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF]
    return int(np.argmax(np.stack(c, 1).reshape(-1)[:vocab] >> np.uint64(9)))


def _forward64(shape, w, tokens, first_row):
    """Logits of rows first_row.. of one sequence in fp64; keys and values are stored as bf16, as the cache does."""
    hd, hq, hkv = shape.head_dim, shape.n_q_heads, shape.n_kv_heads
    n = len(tokens)
    h = w["embed"][torch.tensor(tokens, device="cuda")].double()
    pos = torch.arange(n, device="cuda", dtype=torch.float64)
    inv = shape.rope_theta ** (-2.0 * torch.arange(hd // 2, device="cuda", dtype=torch.float64) / hd)
    cos, sin = torch.cos(pos[:, None] * inv), torch.sin(pos[:, None] * inv)

    def norm(x, gain):
        return x / torch.sqrt((x * x).mean(-1, keepdim=True) + shape.rms_eps) * gain.double()

    def rope(x, first=0):  # [rows][heads][hd], rows from position `first`
        a, b = x[..., :hd // 2], x[..., hd // 2:]
        c, s = cos[first:, None], sin[first:, None]
        return torch.cat([a * c - b * s, b * c + a * s], -1)

    lo = 0
    for l, L in enumerate(w["layers"]):
        x = norm(h, L["attn_norm"])
        k = rope((x @ L["wk"].double().T).view(n, hkv, hd)).to(torch.bfloat16).double()
        v = (x @ L["wv"].double().T).view(n, hkv, hd).to(torch.bfloat16).double()
        if l == shape.n_layers - 1:
            lo = first_row  # the last layer's other rows reach no output
        q = rope((x[lo:] @ L["wq"].double().T).view(n - lo, hq, hd), lo)
        o = torch.empty((n - lo, hq, hd), device="cuda", dtype=torch.float64)
        hide = torch.arange(n, device="cuda")[None, :] > torch.arange(lo, n, device="cuda")[:, None]
        for j in range(hq):
            p = (q[:, j] @ k[:, j * hkv // hq].T) / math.sqrt(hd)
            o[:, j] = torch.softmax(p.masked_fill(hide, -math.inf), -1) @ v[:, j * hkv // hq]
        h = h[lo:] + o.reshape(n - lo, hq * hd) @ L["wo"].double().T
        x = norm(h, L["mlp_norm"])
        g = x @ L["wg"].double().T
        h = h + (g / (1.0 + torch.exp(-g)) * (x @ L["wu"].double().T)) @ L["wd"].double().T
    x = norm(h[first_row - lo:], w["final_norm"])
    out = [x @ w["lm_head"][i:i + 16384].double().T for i in range(0, shape.vocab, 16384)]
    return torch.cat(out, -1)


def exact(case, seed):
    if case["kind"] in ("cod", "accept"):
        return None  # whole numbers
    t, d = _shapes(case)
    shape, mine = (d, 2 * seed + 1) if case["kind"] == "draft" else (t, 2 * seed)
    lens, K = _lens(case), case["K"]
    extra = (K + 1) * max(case["steps"], 1)
    mats = sum(int(np.prod(shape.tensor_shape(k))) for k in S.LAYER_TENSORS)
    if 2.0 * mats * (shape.n_layers - 0.6) * (sum(lens) + extra * len(lens)) > 1.4e13:
        return None  # over 20 seconds
    w = _weights(shape, mine)
    prompts, cand = _prompts(case, seed, t.vocab), _candidates(case, seed, t.vocab).tolist()
    rows = []
    for b, p in enumerate(prompts):
        toks = p + [_philox_argmax(seed, 2, 0, b, 0, t.vocab)]
        if case["kind"] == "draft":
            toks += [d.mask_id] * (K - 1)
        elif case["kind"] == "generate":
            for i in range(case["steps"]):
                toks += [_philox_argmax(seed, 0, i + 1, b, j, t.vocab) for j in range(K)]
                toks += [_philox_argmax(seed, 2, i + 1, b, 0, t.vocab)]
            toks = toks[:-1]
        else:
            toks += cand[b][:K]
        keep = K if case["kind"] == "draft" else K + 1
        rows.append(_forward64(shape, w, toks, len(toks) - keep))
    logits = torch.stack(rows)
    if case["kind"] == "draft":
        return {"draft_logits": logits}
    if case["kind"] == "verify":
        return {"logits": logits}
    if case["kind"] == "prefill":
        return {"first": None, "logits": logits}
    none = [None] * case["steps"]
    return {"first": None, "emitted": none, "accept_len": none, "kv_slots": none, "logits": logits}
