"""The performance cases: passes through the public entry points of the packed-cache
attention step, over the sizes, formats and directions it is used with.

  project   the Q/K/V projection with LoRA branches and RoPE (bf16 or NF4 base): a
            prompt's, or a decode step's of several layers replayed from a captured
            CUDA graph
  append    quantize-and-pack of a prompt's keys and values, whole or in chunks
  prefill   causal attention of a prompt (or its last chunk) over the packed cache
  decode    one decode step's attention over the packed caches of several layers
            (uniform, ragged and paged), replayed from a captured CUDA graph
  generate  a whole call: prompt projection, append, prefill attention, then
            decode steps replayed from a captured CUDA graph
  backward  the straight-through backward of one layer: attention, then adapters

Model shapes are the workloads of `paper_2609_04263_gb300.synth`.
"""
import math

import numpy as np
import torch

from paper_2609_04263_gb300 import api, kvq

DEV = "cuda"

# hidden, query heads, kv heads, head_dim, RoPE base, activations
MODELS = {
    "small_f32": (256, 4, 4, 64, 1e4, torch.float32),
    "tinyllama": (2048, 32, 4, 64, 1e4, torch.bfloat16),
    "llama8b": (4096, 32, 8, 128, 5e5, torch.bfloat16),
    "gemma12b": (3840, 16, 8, 256, 1e4, torch.bfloat16),
}
# format, key bits, value bits, group size, residual tokens, sink tokens
FORMATS = {
    "affine4": (kvq.KVQ_FMT_AFFINE, 4, 4, 32, 0, 0),
    "affine2": (kvq.KVQ_FMT_AFFINE, 2, 2, 32, 0, 0),
    "sym2": (kvq.KVQ_FMT_SYMMETRIC, 2, 2, 32, 0, 0),
    "kivi2": (kvq.KVQ_FMT_KIVI, 2, 2, 32, 128, 0),
    "kvarn": (kvq.KVQ_FMT_KVARN, 4, 2, 64, 0, 128),
}
NORM_ITERS = 8
ALPHA_OVER_R = 2.0
PLANES = ("k_codes", "k_scale", "k_zero", "v_codes", "v_scale", "v_zero", "k_full", "v_full",
          "k_pend", "v_pend", "k_row", "k_col", "v_row", "v_col")


def listed():
    return [
        # the smallest model: one fp32 layer, a 512-token prompt, then 64 decode steps
        dict(name="generate_small_f32", op="generate", model="small_f32", fmt="affine4", layers=1,
             batch=1, prompt=512, steps=64, rank=8),
        # a decode step's projections of a 16-sequence batch: each layer's weights are read once
        dict(name="project_decode_8b", op="project", model="llama8b", base="bf16", layers=4,
             batch=16, length=1, rank=16),
        # the projection of a batch of prompts
        dict(name="project_prompt_8b", op="project", model="llama8b", base="bf16", layers=1,
             batch=4, length=2048, rank=16),
        # a calibration sequence through an NF4 base
        dict(name="project_nf4_8b", op="project", model="llama8b", base="nf4", layers=1, batch=1,
             length=2048, rank=16),
        # quantize-and-pack of long prompts, with the Hadamard rotation and normalisation
        dict(name="append_kvarn_12b", op="append", model="gemma12b", fmt="kvarn", batch=4,
             length=8000, chunk=0),
        # prompt attention, small heads, a batch of ragged-sized prompts
        dict(name="prefill_affine4_tinyllama", op="prefill", model="tinyllama", fmt="affine4",
             batch=4, tokens=2029, length=2029),
        # the largest prompt attention of the default benchmark's shape
        dict(name="prefill_kivi2_8b", op="prefill", model="llama8b", fmt="kivi2", batch=2,
             tokens=8192, length=8192),
        # long-prompt attention at head_dim 256
        dict(name="prefill_kvarn_12b", op="prefill", model="gemma12b", fmt="kvarn", batch=1,
             tokens=8192, length=8192),
        # decode attention of a 16-sequence batch at long context
        dict(name="decode_kivi2_8b", op="decode", model="llama8b", fmt="kivi2", layers=4,
             batch=16, tokens=8201, layout="uniform"),
        dict(name="decode_kvarn_12b", op="decode", model="gemma12b", fmt="kvarn", layers=4,
             batch=4, tokens=8300, layout="uniform"),
        # a served request batch on the small model: prompt, then decode steps
        dict(name="generate_tinyllama", op="generate", model="tinyllama", fmt="affine4", layers=4,
             batch=4, prompt=1000, steps=32, rank=16),
        # one calibration step's backward of a layer over a 1000-token sequence
        dict(name="backward_kivi2_8b", op="backward", model="llama8b", fmt="kivi2", batch=1,
             length=1000, rank=16),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(("project", "append", "prefill", "decode", "generate", "backward"))
    if op == "project":
        base = rng.choice(("bf16", "bf16", "nf4"))
        model = "llama8b" if base == "nf4" else rng.choice(("tinyllama", "llama8b", "gemma12b"))
        layers = 1
        if rng.random() < 0.5:
            batch, length, layers = _log(rng, 1, 16), 1, 4
        else:
            length = _log(rng, 17, 8192)
            batch = max(1, min(_log(rng, 1, 16), 8192 // length))
        return dict(op=op, model=model, base=base, layers=layers, batch=batch, length=length,
                    rank=rng.choice((8, 16, 32, 64)))
    if op == "append":
        fmt = rng.choice(("affine4", "sym2", "kivi2", "kvarn"))
        model = {"kivi2": "llama8b", "kvarn": "gemma12b"}.get(fmt, "tinyllama")
        length = _log(rng, 16, 8192)
        batch = max(1, min(_log(rng, 1, 16), 32768 // length))
        chunk = rng.choice((0, 128, 512))
        return dict(op=op, model=model, fmt=fmt, batch=batch, length=length,
                    chunk=0 if chunk >= length or length > 16 * chunk else chunk)
    if op == "prefill":
        fmt, model = rng.choice((("affine4", "tinyllama"), ("sym2", "tinyllama"),
                                 ("kivi2", "llama8b"), ("affine2", "llama8b"),
                                 ("kvarn", "gemma12b")))
        tokens = _log(rng, 16, 8192)
        most = max(1, int((8192 / tokens) ** 2)) * (1 if fmt == "kvarn" else 2)
        batch = min(_log(rng, 1, 8), most, max(1, 16384 // tokens))
        length = tokens if rng.random() < 0.7 else min(tokens, 128)
        return dict(op=op, model=model, fmt=fmt, batch=batch, tokens=tokens, length=length)
    if op == "decode":
        fmt, model = rng.choice((("affine4", "tinyllama"), ("sym2", "tinyllama"),
                                 ("kivi2", "llama8b"), ("affine4", "llama8b"),
                                 ("kvarn", "gemma12b")))
        layout = "uniform" if fmt == "kvarn" else rng.choice(("uniform", "ragged", "paged"))
        tokens = _log(rng, 64, 8300)
        batch = max(1, min(_log(rng, 1, 16), 131072 // tokens))
        return dict(op=op, model=model, fmt=fmt, layers=rng.choice((2, 4)), batch=batch,
                    tokens=tokens, layout=layout)
    if op == "generate":
        model, fmt, rank = rng.choice((("small_f32", "affine4", 8), ("tinyllama", "affine4", 16),
                                       ("tinyllama", "sym2", 64), ("llama8b", "kivi2", 16),
                                       ("gemma12b", "kvarn", 32)))
        prompt = _log(rng, 17, {"small_f32": 600, "gemma12b": 1024}.get(model, 2048))
        batch = 1 if model == "small_f32" else max(1, min(_log(rng, 1, 8), 4096 // prompt))
        return dict(op=op, model=model, fmt=fmt, layers=1 if model == "small_f32" else 2,
                    batch=batch, prompt=prompt, steps=rng.choice((8, 16, 32)), rank=rank)
    model, fmt = rng.choice((("tinyllama", "affine4"), ("tinyllama", "sym2"),
                             ("llama8b", "kivi2"), ("llama8b", "affine2")))
    return dict(op=op, model=model, fmt=fmt, batch=1, length=_log(rng, 32, 1200),
                rank=rng.choice((8, 16, 32)))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
class _Rand:
    """Seeded draws on the device."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV).manual_seed(int(seed))

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device=DEV)

    def kv(self, B, H, L, D, dtype):
        """Keys or values: every channel with its own scale in [1/2, 2] and offset."""
        scale = torch.exp2(2.0 * torch.rand(D, generator=self.g, device=DEV) - 1.0)
        return (self.normal(B, H, L, D) * scale + 0.25 * self.normal(D)).to(dtype).contiguous()

    def hidden(self, model, *shape):
        """Hidden states: heavy tails (Student-t, 4 degrees of freedom) for the
        12B-class shape, else N(0, 1) with 1% of the channels scaled x20 in bf16;
        at unit RMS, as the norm before a model's attention leaves them."""
        x = self.normal(*shape)
        if model == "gemma12b":
            x = x * torch.rsqrt(sum(self.normal(*shape) ** 2 for _ in range(4)) / 4.0)
        elif model != "small_f32":
            d = shape[-1]
            x[..., torch.randperm(d, generator=self.g, device=DEV)[:d // 100]] *= 20.0
        return (x * torch.rsqrt(x.square().mean(-1, True))).to(MODELS[model][5])

    def weights(self, model, rank, base="bf16"):
        d_in, hq, hkv, D, _, dt = MODELS[model]
        n = (hq + 2 * hkv) * D
        if base == "nf4":
            codes = torch.randint(0, 256, (n, d_in // 2), generator=self.g, device=DEV,
                                  dtype=torch.uint8)
            absmax = (0.02 * self.normal(n, d_in // 64, 64)).abs().amax(-1).contiguous()
            w = (codes, absmax)
        else:
            w = (0.02 * self.normal(n, d_in)).to(dt)
        lora = {p: ((0.02 * self.normal(rank, d_in)).to(dt),
                    (0.01 * self.normal(h * D, rank)).to(dt))
                for p, h in (("q", hq), ("k", hkv), ("v", hkv))}
        return w, lora


def _cache(case, max_tokens, layout="uniform", num_pages=0):
    _, hq, hkv, D, _, dt = MODELS[case["model"]]
    fmt, kb, vb, G, R, S = FORMATS[case["fmt"]]
    desc = api.make_desc(fmt, kb, vb, G, case["batch"], hkv, hq, D, max_tokens, dt,
                         residual_tokens=R, sink_tokens=S, norm_iters=NORM_ITERS,
                         layout={"uniform": kvq.KVQ_LAYOUT_UNIFORM,
                                 "ragged": kvq.KVQ_LAYOUT_RAGGED,
                                 "paged": kvq.KVQ_LAYOUT_PAGED}[layout], num_pages=num_pages)
    return api.Cache(desc, buffer=torch.zeros(kvq.kvq_cache_bytes(desc), dtype=torch.uint8,
                                              device=DEV))


def _planes(cache):
    """The cache's planes as tensors (views of its buffer)."""
    p = cache.planes()
    return {k: p[k] for k in PLANES if k in p}


def _lengths(case):
    """Tokens of each sequence of a decode batch."""
    B, T = case["batch"], case["tokens"]
    if case["layout"] == "uniform":
        return [T] * B
    return [T - (T // 2) * b // max(B - 1, 1) for b in range(B)]


def _captured(fn):
    """fn's launches as a CUDA graph, captured on a side stream."""
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        fn()
    torch.cuda.synchronize()
    return g


def _inputs(case, seed):
    """The tensors a pass starts from."""
    op, model = case["op"], case["model"]
    d_in, hq, hkv, D, _, dt = MODELS[model]
    B, r = case["batch"], _Rand(seed)
    i = {}
    if op == "project":
        i["layers"] = [r.weights(model, case["rank"], case["base"]) for _ in range(case["layers"])]
        i["x"] = r.hidden(model, B, case["length"], d_in)
    elif op == "append":
        i["k"], i["v"] = (r.kv(B, hkv, case["length"], D, dt) for _ in range(2))
    elif op == "prefill":
        i["k"], i["v"] = (r.kv(B, hkv, case["tokens"], D, dt) for _ in range(2))
        i["q"] = r.normal(B, hq, case["length"], D).to(dt)
    elif op == "decode":
        i["kv"] = [tuple(r.kv(B, hkv, case["tokens"], D, dt) for _ in range(2))
                   for _ in range(case["layers"])]
        i["q"] = [r.normal(B, hq, 1, D).to(dt) for _ in range(case["layers"])]
    elif op == "generate":
        i["layers"] = [r.weights(model, case["rank"]) for _ in range(case["layers"])]
        x = r.hidden(model, B, case["prompt"] + case["steps"], d_in)
        i["x"] = x[:, :case["prompt"]].contiguous()
        i["x_dec"] = x[:, case["prompt"]:].transpose(0, 1).unsqueeze(2).contiguous()
    else:
        L = case["length"]
        i["w"], i["lora"] = r.weights(model, case["rank"])
        i["x"] = r.hidden(model, B, L, d_in)
        i["k"], i["v"] = (r.kv(B, hkv, L, D, dt) for _ in range(2))
        i["q"], i["d_out"] = (r.normal(B, hq, L, D).to(dt) for _ in range(2))
    return i


def prepare(case, seed):
    op = case["op"]
    s = {"case": case, **_inputs(case, seed)}
    if op == "project" and case["length"] == 1:
        _, hq, hkv, D, _, dt = MODELS[case["model"]]
        s["out"] = [tuple(torch.empty(case["batch"], h, 1, D, dtype=dt, device=DEV)
                          for h in (hq, hkv, hkv)) for _ in s["layers"]]
        _project(s)
        s["graph"] = _captured(lambda: _project(s))
    elif op == "append":
        s["cache"] = _cache(case, case["length"])
        c = case["chunk"] or case["length"]
        s["chunks"] = [(s["k"][:, :, t:t + c].contiguous(), s["v"][:, :, t:t + c].contiguous())
                       for t in range(0, case["length"], c)]
        s["planes"] = _planes(s["cache"])
    elif op in ("prefill", "backward"):
        s["cache"] = _cache(case, s["k"].shape[2])
        s["cache"].append(s["k"], s["v"])
    elif op == "decode":
        _prepare_decode(s)
    elif op == "generate":
        _prepare_generate(s)
    return s


def _prepare_decode(s):
    case = s["case"]
    lens = _lengths(case)
    pages = sum((t + kvq.KVQ_PAGE_TOKENS - 1) // kvq.KVQ_PAGE_TOKENS for t in lens)
    s["caches"] = []
    for k, v in s["kv"]:
        c = _cache(case, case["tokens"] + 64, case["layout"], pages)
        if case["layout"] == "uniform":
            c.append(k, v)
        else:
            c.append_ragged(k, v, lens)
        s["caches"].append(c)
    s["out"] = [torch.empty_like(q) for q in s["q"]]

    def step():
        for c, q, o in zip(s["caches"], s["q"], s["out"]):
            c.attend_decode(q, out=o)

    step()
    s["graph"] = _captured(step)
    del s["kv"]


def _prepare_generate(s):
    case = s["case"]
    _, hq, hkv, D, base, dt = MODELS[case["model"]]
    B, n, layers = case["batch"], case["steps"], case["layers"]
    s["caches"] = [_cache(case, case["prompt"] + n) for _ in range(layers)]
    s["fused"] = s["caches"][0].project_append_supported(
        case["prompt"], s["x"].shape[-1], s["layers"][0][1])
    s["outs"] = torch.zeros(n, layers, B, hq, 1, D, dtype=dt, device=DEV)
    one = lambda h: torch.empty(B, h, 1, D, dtype=dt, device=DEV)
    qkv = (one(hq), one(hkv), one(hkv))
    s["o_step"] = torch.empty(layers, B, hq, 1, D, dtype=dt, device=DEV)
    s["x_step"] = torch.empty_like(s["x_dec"][0])
    s["steps"] = [(s["x_dec"][t], s["outs"][t]) for t in range(n)]

    def step():
        for c, (w, lora), o in zip(s["caches"], s["layers"], s["o_step"]):
            c.decode_step(s["x_step"], w, lora, ALPHA_OVER_R, base, qkv=qkv, out=o)

    _prompt(s)
    s["graph"] = _captured(step)
    s["planes"] = [_planes(c) for c in s["caches"]]
    s["qkv"] = qkv


def _prompt(s):
    """Every layer's prompt: projection, append, prefill attention."""
    _, hq, hkv, D, base, _ = MODELS[s["case"]["model"]]
    outs = []
    for c, (w, lora) in zip(s["caches"], s["layers"]):
        c.reset()
        if s["fused"]:
            q = c.project_append(s["x"], w, lora, ALPHA_OVER_R, base)
        else:
            q, k, v = api.project_lora(s["x"], w, lora, ALPHA_OVER_R, hq, hkv, D, rope_base=base)
            c.append(k, v)
        outs.append(c.attend_prefill(q))
    return outs


def _project(s):
    """Every layer's projection of the same hidden states, at positions from 100."""
    case = s["case"]
    _, hq, hkv, D, base, _ = MODELS[case["model"]]
    outs = s.get("out") or [None] * case["layers"]
    if case["base"] == "nf4":
        return [api.project_lora_nf4(s["x"], *w, lora, ALPHA_OVER_R, hq, hkv, D, pos0=100,
                                     rope_base=base, out=o)
                for (w, lora), o in zip(s["layers"], outs)]
    return [api.project_lora(s["x"], w, lora, ALPHA_OVER_R, hq, hkv, D, pos0=100, rope_base=base,
                             out=o) for (w, lora), o in zip(s["layers"], outs)]


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    case = s["case"]
    op = case["op"]
    _, hq, hkv, D, base, _ = MODELS[case["model"]]
    if op == "project":
        if "graph" not in s:
            return _project(s)
        s["graph"].replay()
        return s["out"]
    if op == "append":
        s["cache"].reset()
        for k, v in s["chunks"]:
            s["cache"].append(k, v)
        return s["planes"]
    if op == "prefill":
        return s["cache"].attend_prefill(s["q"])
    if op == "decode":
        s["graph"].replay()
        return s["out"]
    if op == "generate":
        prompt = _prompt(s)
        for x, o in s["steps"]:
            s["x_step"].copy_(x)
            s["graph"].replay()
            o.copy_(s["o_step"])
        return {"prompt": prompt, "steps": s["outs"], "caches": s["planes"]}
    dq, dk, dv = s["cache"].attend_backward(s["q"], s["d_out"])
    grads, dx = api.lora_backward(s["x"], s["w"], s["lora"], ALPHA_OVER_R, hq, hkv, D, dq, dk, dv,
                                  rope_base=base, want_dx=True)
    return {"dq": dq, "dk": dk, "dv": dv, "adapters": grads, "dx": dx}


# ---------------------------------------------------------------------------
# what a pass cannot do without, and how far another correct one may be off
# ---------------------------------------------------------------------------
def _cache_bytes(case, tokens):
    """Bytes that one (sequence, kv head) of a cache holds for `tokens` tokens."""
    D, dt = MODELS[case["model"]][3], MODELS[case["model"]][5]
    fmt, kb, vb, G, R, S = FORMATS[case["fmt"]]
    act = 4 if dt == torch.float32 else 2
    code = D * (kb + vb) // 8
    per_group = 2 * D // G
    if fmt == kvq.KVQ_FMT_AFFINE:
        return tokens * (code + 4 * per_group)
    if fmt == kvq.KVQ_FMT_SYMMETRIC:
        return tokens * (code + 2 * per_group)
    if fmt == kvq.KVQ_FMT_KIVI:
        coded = max(0, tokens - R) // G * G
        return coded * (code + 2 * per_group) + coded // G * 4 * D + (tokens - coded) * 2 * D * act
    coded = max(0, tokens - S) // G * G
    return coded * (code + 4 * per_group + 4) + coded // G * 4 * D + (tokens - coded) * 2 * D * act


def work(case):
    op = case["op"]
    d_in, hq, hkv, D, _, dt = MODELS[case["model"]]
    act = 4 if dt == torch.float32 else 2
    B, n = case["batch"], (hq + 2 * hkv) * D

    def project(rows, rank, weight_bytes):
        return (rows * (d_in + n) * act + weight_bytes + rank * (3 * d_in + n) * act,
                2 * rows * (n * d_in + rank * (3 * d_in + n)))

    def attend(length, tokens):
        seen = length * tokens - length * (length - 1) // 2
        return (2 * B * hq * length * D * act + B * hkv * _cache_bytes(case, tokens),
                4 * B * hq * seen * D)

    if op == "project":
        wb = n * d_in * 9 // 16 if case["base"] == "nf4" else n * d_in * act
        b, f = (case["layers"] * t for t in project(B * case["length"], case["rank"], wb))
    elif op == "append":
        b = 2 * B * hkv * case["length"] * D * act + B * hkv * _cache_bytes(case, case["length"])
        f = 0
    elif op == "prefill":
        b, f = attend(case["length"], case["tokens"])
    elif op == "decode":
        got = [hkv * _cache_bytes(case, t) + 2 * hq * D * act for t in _lengths(case)]
        b, f = case["layers"] * sum(got), case["layers"] * 4 * hq * D * sum(_lengths(case))
    elif op == "generate":
        P, N, wb = case["prompt"], case["steps"], n * d_in * act
        parts = [project(B * P, case["rank"], wb), attend(P, P)]
        for t in range(N):
            parts += [project(B, case["rank"], wb), attend(1, P + t + 1)]
        b, f = (case["layers"] * sum(p[i] for p in parts) for i in (0, 1))
    else:
        L, r = case["length"], case["rank"]
        pairs = L * (L + 1) // 2
        b = (2 * B * hq * L * D * act + B * hkv * _cache_bytes(case, L)          # q, d_out, cache
             + (B * hq + 2 * B * hkv) * L * D * 4 + B * L * d_in * (act + 4)     # dq dk dv, x dx
             + n * d_in * act + r * (3 * d_in + n) * (act + 4))                  # W, factors
        f = 10 * B * hq * pairs * D + 2 * B * L * n * d_in + 8 * B * L * r * (3 * d_in + n)
    return {"bytes": b, "flops": f}


def tolerance(case):
    # about four times what the path is off from exact(), below
    op = case["op"]
    if op == "append":
        return "exact"
    if op == "project":
        return {"rel": 8e-3, "max": 4e-2}
    if op == "prefill":
        return {"rel": 7e-3, "max": 3e-2}
    if op == "decode":
        # long contexts average the values to small outputs
        if case["fmt"] == "kvarn":
            return {"rel": 7e-3, "max": 3e-2}
        return {"rel": 3e-2, "max": 0.12}
    if op == "backward":
        # fp32 sums; dx multiplies gradients split in two bf16 parts
        return {"rel": 7e-5, "max": 3e-4}
    # a key or value that rounds the other way in the projection now and then moves its code
    if MODELS[case["model"]][5] == torch.float32:
        return {"rel": 4e-4, "max": 2e-3, "differ": 1e-4}
    return {"rel": 3e-2, "max": 0.99, "differ": 2e-3}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _rope(y, pos, base, back=False):
    half = y.shape[-1] // 2
    i = torch.arange(half, dtype=torch.float64, device=DEV)
    ang = pos.double()[:, None] * base ** (-i / half)[None]
    c, s = torch.cos(ang), torch.sin(ang) * (-1.0 if back else 1.0)
    a, b = y[..., :half], y[..., half:]
    return torch.cat([a * c - b * s, b * c + a * s], -1)


def _nf4_levels():
    """QLoRA's NormalFloat levels: quantiles of N(0, 1), 8 positive and 7 negative
    ones and 0, scaled to 1."""
    delta = 0.5 * (1.0 / 30.0 + 1.0 / 32.0)
    ppf = lambda p: torch.special.ndtri(torch.tensor(p, dtype=torch.float64))
    pos = ppf(np.linspace(1.0 - delta, 0.5, 9)[:-1].tolist())
    neg = -ppf(np.linspace(1.0 - delta, 0.5, 8)[:-1].tolist())
    v = torch.cat([pos, neg, torch.zeros(1, dtype=torch.float64)]).sort().values
    return (v / v.abs().max()).to(DEV)


def _project64(model, x, w, lora, pos0=0):
    d_in, hq, hkv, D, base, _ = MODELS[model]
    if isinstance(w, tuple):
        codes, absmax = w
        idx = torch.stack([codes & 15, codes >> 4], -1).reshape(codes.shape[0], d_in).long()
        w = _nf4_levels()[idx] * absmax.double().repeat_interleave(64, 1)
    B, L, _ = x.shape
    x = x.double().reshape(B * L, d_in)
    pos = pos0 + torch.arange(L, device=DEV)
    outs, lo = [], 0
    for p, h in (("q", hq), ("k", hkv), ("v", hkv)):
        a, b = (t.double() for t in lora[p])
        y = x @ w[lo:lo + h * D].double().T + ALPHA_OVER_R * ((x @ a.T) @ b.T)
        lo += h * D
        y = y.reshape(B, L, h, D).transpose(1, 2)
        outs.append(_rope(y, pos, base) if p in "qk" else y)
    return outs


def _over(x, q):
    """x / q, rounded once (division by a plain number multiplies by its reciprocal)."""
    return x / torch.full_like(x, q)


def _affine(x, bits):
    """Codes, fp16 scale and fp16 offset of the groups on the last axis (codes and
    metadata are defined in fp32)."""
    x, q = x.float(), 2 ** bits - 1
    mn, mx = x.amin(-1, True), x.amax(-1, True)
    s = torch.clamp(_over(mx - mn, q), min=1e-8)
    return torch.clamp(torch.round((x - mn) / s), 0, q), s.half(), (mn + 0.0).half()


def _grouped(x, bits, G, fmt):
    """The reconstruction of x after coding in groups of G on the last axis."""
    y = x.reshape(*x.shape[:-1], -1, G)
    if fmt == kvq.KVQ_FMT_SYMMETRIC:
        q = 2 ** (bits - 1) - 1
        s = torch.clamp(_over(y.float().abs().amax(-1, True), q), min=1e-8)
        r = torch.clamp(torch.round(y.float() / s), -q, q).double() * s.half().double()
    else:
        c, s, m = _affine(y, bits)
        r = c.double() * s.double() + m.double()
    return r.reshape(x.shape)


def _hadamard(D):
    h = torch.ones(1, 1, dtype=torch.float64, device=DEV)
    while h.shape[0] < D:
        h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)])
    return h / math.sqrt(D)


def _kvarn_block(y):
    """Rows and columns of rotated blocks y [..., G, D] brought to unit RMS in turn."""
    r, c = torch.ones_like(y[..., :1]), torch.ones_like(y[..., :1, :])
    for _ in range(NORM_ITERS):
        s = y.square().mean(-1, True).sqrt().clamp(min=1e-8)
        y, r = y / s, r * s
        s = y.square().mean(-2, True).sqrt().clamp(min=1e-8)
        y, c = y / s, c * s
    return y, r.half().double(), c.half().double()


def _reconstruct(case, k, v):
    """What a cache holding k, v [B, H, T, D] gives attention, in 64 bits."""
    fmt, kb, vb, G, R, S = FORMATS[case["fmt"]]
    T, D = k.shape[2:]
    if fmt in (kvq.KVQ_FMT_AFFINE, kvq.KVQ_FMT_SYMMETRIC):
        return _grouped(k, kb, G, fmt), _grouped(v, vb, G, fmt)
    if fmt == kvq.KVQ_FMT_KIVI:
        n = max(0, T - R) // G * G
        kq, vq = k[:, :, :n], v[:, :, :n]
        if n:
            t = kq.reshape(*kq.shape[:2], n // G, G, D).transpose(-1, -2)
            kq = _grouped(t, kb, G, fmt).transpose(-1, -2).reshape(kq.shape)
            vq = _grouped(vq, vb, G, fmt)
        return (torch.cat([kq.double(), k[:, :, n:].double()], 2),
                torch.cat([vq.double(), v[:, :, n:].double()], 2))
    n = max(0, T - S) // G * G
    got = []
    for x, bits in ((k, kb), (v, vb)):
        x = x.double()
        if n:
            h = _hadamard(D)
            y, r, c = _kvarn_block((x[:, :, S:S + n] @ h).reshape(*x.shape[:2], n // G, G, D))
            y = (_grouped(y, bits, G, kvq.KVQ_FMT_AFFINE) * r * c).reshape(*x.shape[:2], n, D) @ h
            x = torch.cat([x[:, :, :S], y, x[:, :, S + n:]], 2)
        got.append(x)
    return got


def _attend64(q, k, v, lens=None):
    """Causal attention of the newest q.shape[2] tokens (of each sequence's lens)."""
    B, hq, L, D = q.shape
    g = hq // k.shape[1]
    out = torch.empty(q.shape, dtype=torch.float64, device=DEV)
    for b in range(B):
        T = k.shape[2] if lens is None else lens[b]
        for h in range(hq):
            for lo in range(0, L, 2048):
                hi = min(L, lo + 2048)
                n = T - L + hi
                s = q[b, h, lo:hi].double() @ k[b, h // g, :n].T / math.sqrt(D)
                seen = torch.arange(n, device=DEV)[None] <= (
                    T - L + torch.arange(lo, hi, device=DEV))[:, None]
                s.masked_fill_(~seen, -math.inf)
                out[b, h, lo:hi] = torch.softmax(s, -1) @ v[b, h // g, :n]
    return out


def _exact_generate(case, i):
    P, N = case["prompt"], case["steps"]
    model = case["model"]
    dt = MODELS[model][5]
    x = torch.cat([i["x"], i["x_dec"].squeeze(2).transpose(0, 1)], 1)
    prompts, steps = [], []
    for w, lora in i["layers"]:
        # queries, keys and values leave the projection in the activations' type
        q, k, v = (t.to(dt) for t in _project64(model, x, w, lora))
        got = []
        for T in [P] + list(range(P + 1, P + N + 1)):
            rk, rv = _reconstruct(case, k[:, :, :T], v[:, :, :T])
            got.append(_attend64(q[:, :, :P] if T == P else q[:, :, T - 1:T], rk, rv))
        prompts.append(got[0])
        steps.append(torch.stack(got[1:]))
    return {"prompt": prompts, "steps": torch.stack(steps, 1), "caches": None}


def _exact_backward(case, i):
    _, hq, hkv, D, base, _ = MODELS[case["model"]]
    B, L, g = case["batch"], case["length"], hq // hkv
    k, v = _reconstruct(case, i["k"], i["v"])
    q, do, sc = i["q"].double(), i["d_out"].double(), 1.0 / math.sqrt(D)
    dq, dk, dv = torch.zeros_like(q), torch.zeros_like(k), torch.zeros_like(v)
    mask = torch.ones(L, L, dtype=torch.bool, device=DEV).triu(1)
    for b in range(B):
        for h in range(hq):
            K, V = k[b, h // g], v[b, h // g]
            p = torch.softmax((q[b, h] @ K.T * sc).masked_fill(mask, -math.inf), -1)
            dv[b, h // g] += p.T @ do[b, h]
            dp = do[b, h] @ V.T
            ds = p * (dp - (p * dp).sum(-1, True)) * sc
            dq[b, h] = ds @ K
            dk[b, h // g] += ds.T @ q[b, h]
    pos = torch.arange(L, device=DEV)
    x, w = i["x"].double().reshape(B * L, -1), i["w"].double()
    dx, grads, lo = 0.0, {}, 0
    for p, y in (("q", _rope(dq, pos, base, True)), ("k", _rope(dk, pos, base, True)), ("v", dv)):
        y = y.transpose(1, 2).reshape(B * L, -1)
        a, bm = (t.double() for t in i["lora"][p])
        u = ALPHA_OVER_R * (y @ bm)
        grads[p] = (u.T @ x, ALPHA_OVER_R * (y.T @ (x @ a.T)))
        dx = dx + y @ w[lo:lo + y.shape[1]] + u @ a
        lo += y.shape[1]
    return {"dq": dq, "dk": dk, "dv": dv, "adapters": grads, "dx": dx.reshape(i["x"].shape)}


def exact(case, seed):
    op = case["op"]
    i = _inputs(case, seed)
    if op == "project":
        return [_project64(case["model"], i["x"], w, lora, 100) for w, lora in i["layers"]]
    if op == "append":
        return None            # codes and their metadata are compared bit for bit
    if op == "prefill":
        return _attend64(i["q"], *_reconstruct(case, i["k"], i["v"]))
    if op == "decode":
        lens = _lengths(case)
        got = []
        for (k, v), q in zip(i["kv"], i["q"]):
            one = []
            for b, T in enumerate(lens):
                rk, rv = _reconstruct(case, k[b:b + 1, :, :T], v[b:b + 1, :, :T])
                one.append(_attend64(q[b:b + 1], rk, rv))
            got.append(torch.cat(one))
        return got
    return _exact_generate(case, i) if op == "generate" else _exact_backward(case, i)
