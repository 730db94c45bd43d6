"""The measured work of this library: what a serving loop has it do on one
GPU, through the public binding (``paper_2608_15171_gb300.ppas``).

Two kinds of pass:

* ``step``: the attention part of one scheduler iteration over ``layers``
  layers, each with its own paged cache: ``ppas_kv_append`` of the new
  tokens' keys and values, then ``ppas_attention_step`` (or its no-allocation
  form) of the iteration's rows, decode rows first, then prefill chunks.  The
  plan of such a pass (lengths, block tables, slots) and the workspace are
  what the loop holds when it reaches the layers.  Iterations of few rows run
  several layers a pass, so that a pass streams its K/V from memory and not
  from the cache of the pass before.
* ``gateup``: the gate-up projection of the decoder MLP over the iteration's
  tokens (``ppas_gateup_swiglu``, weights packed once).

Sizes are those of the repository's workloads (Qwen2.5-3B and Llama-3.1-8B
attention geometries, 16-token pages in random order, the 2k and 16k token
budgets, 20k-30k contexts, the 4 x 512 tiny workload); ``draw`` spreads over
the ranges between and around them.
"""
import math

import numpy as np
import torch

from paper_2608_15171_gb300 import ppas

PAGE = 16
DIM = 128


# ------------------------------------------------------------------ the cases
def _step(name, hq, hk, decodes=0, dec_lo=1, dec_hi=1, chunks="", pre_lo=0, pre_hi=0, lens_seed=0, layers=1,
          fp32=False, entry="workspace", gain=1.0):
    return {"name": name, "kind": "step", "hq": hq, "hk": hk, "decodes": decodes, "dec_lo": dec_lo, "dec_hi": dec_hi,
            "chunks": chunks, "pre_lo": pre_lo, "pre_hi": pre_hi, "lens_seed": lens_seed, "layers": layers,
            "fp32": fp32, "entry": entry, "gain": gain}


def _gateup(name, tokens, hidden, inter):
    return {"name": name, "kind": "gateup", "tokens": tokens, "hidden": hidden, "inter": inter}


def listed():
    return [
        # one user left, deep in its answer: the smallest iteration a loop runs, bound by latency
        _step("decode 1 x 25k", 16, 2, 1, 25000, 25032, lens_seed=1, layers=8),
        # the usual decode-only iteration of the burst replay
        _step("decode 8 x 25k", 16, 2, 8, 20000, 30064, lens_seed=2, layers=4),
        # a larger GQA model's decode batch: 2 GB of K/V a layer
        _step("decode 16 x 30k", 32, 8, 16, 30000, 30064, lens_seed=3),
        # many short conversations, every length different
        _step("decode 96 x 17-4100", 32, 8, 96, 17, 4100, lens_seed=4, layers=2),
        # the tiny workload's last step: the final 512-token chunk of a prompt beside 2 decodes, fp32 output
        _step("chunk 512 + 2 decodes", 16, 2, 2, 2048, 2048, "512", 1536, 1536, layers=8, fp32=True),
        # prefill pressure under the 2k budget: 4 prompts in progress, 8 decodes
        _step("2k budget, 4 x 512 + 8", 16, 2, 8, 25000, 25031, "512,512,512,512", 0, 24575, lens_seed=5),
        # the same budget on the larger model: 3 ragged chunks, 16 decodes
        _step("2k budget, 3 x 683 + 16", 32, 8, 16, 30000, 30063, "683,683,682", 0, 29317, lens_seed=6),
        # a prompt's first 16k chunk, and what is left of it over the prefix
        _step("chunk 16384", 16, 2, chunks="16384"),
        _step("chunk 8616 over 16384", 16, 2, chunks="8616", pre_lo=16384, pre_hi=16384),
        # the MLP of a decode iteration, of a 2k iteration with 8 decodes, of a 16k chunk
        _gateup("gate-up 8 tokens", 8, 2048, 11008),
        _gateup("gate-up 2056 tokens", 2056, 2048, 11008),
        _gateup("gate-up 16384 tokens", 16384, 2048, 11008),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    if rng.random() < 0.25:
        hidden, inter = rng.choice([(2048, 11008), (2048, 11008), (4096, 14336), (1024, 2816), (1536, 8960)])
        most = min(16384, int(16384 * (2048 * 11008) / (hidden * inter)))
        c = _gateup("", _log_int(rng, 1, most), hidden, inter)
        del c["name"]
        return c
    while True:
        hq, hk = rng.choice([(16, 2), (16, 2), (32, 8), (32, 8), (8, 4), (8, 8)])
        form = rng.choice(["decode", "mixed", "mixed", "prefill"])
        c = _step("", hq, hk, lens_seed=rng.randrange(1 << 20), fp32=rng.random() < 0.2,
                  entry="noalloc" if rng.random() < 0.15 else "workspace", gain=rng.choice([1.0, 1.0, 2.0, 4.0]))
        if form != "prefill":
            c["decodes"] = _log_int(rng, 1, 128)
            c["dec_lo"] = _log_int(rng, 16, 32000)
            c["dec_hi"] = c["dec_lo"] + rng.randrange(c["dec_lo"])
        if form != "decode":
            n = rng.randint(1, 5)
            budget = _log_int(rng, 16 * n, 16384)
            cuts = sorted(rng.sample(range(1, budget), n - 1)) if n > 1 else []
            lens = [b - a for a, b in zip([0] + cuts, cuts + [budget])]
            c["chunks"] = ",".join(str(max(2, x)) for x in lens)
            c["pre_hi"] = rng.choice([0, _log_int(rng, 1, 30000)])
        del c["name"]
        q, k = _lens(c)
        kv = sum(k) * hk * DIM * 4
        c["layers"] = max(1, min(8, int(256e6 // max(kv, 1))))
        if kv <= 2.0e9 and work(c)["flops"] <= 1.4e12 and sum(q) <= 16384 + 128:
            return c


def _lens(case):
    """(q_lens, ctx_lens) of a step: decode rows first."""
    r = np.random.default_rng(case["lens_seed"])
    q = [1] * case["decodes"]
    ctx = [int(x) for x in r.integers(case["dec_lo"], case["dec_hi"] + 1, size=case["decodes"])]
    for n in (int(x) for x in case["chunks"].split(",") if x):
        q.append(n)
        ctx.append(n + int(r.integers(case["pre_lo"], case["pre_hi"] + 1)))
    return q, ctx


# ------------------------------------------------------------------ inputs
def _normal(shape, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).to(torch.bfloat16)


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "gateup":
        t, h, i = case["tokens"], case["hidden"], case["inter"]
        s["x"] = _normal((t, h), seed * 16 + 1)
        # weights of unit-variance products
        s["w"] = (_normal((2 * i, h), seed * 16 + 2).float() / math.sqrt(h)).to(torch.bfloat16)
        s["packed"] = torch.empty_like(s["w"])
        ppas.ppas_gateup_pack(s["w"], s["packed"], h, i)
        s["y"] = torch.empty((t, i), dtype=torch.bfloat16, device="cuda")
        s["err"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        return s
    hq, hk = case["hq"], case["hk"]
    q, ctx = _lens(case)
    rng = np.random.default_rng(seed)
    need = [-(-c // PAGE) for c in ctx]
    s["blocks"] = sum(need) + 8
    order = rng.permutation(s["blocks"]).astype(np.int32)
    table = np.full((len(q), max(need)), -1, np.int32)
    slots, at = [], 0
    for r, (n, nq, c) in enumerate(zip(need, q, ctx)):
        table[r, :n] = order[at:at + n]
        at += n
        pos = np.arange(c - nq, c)
        slots.append(table[r][pos // PAGE] * PAGE + pos % PAGE)
    s["q_lens"], s["ctx_lens"] = np.array(q, np.int32), np.array(ctx, np.int32)
    s["table_host"], s["width"], s["tokens"] = table, max(need), sum(q)
    s["table"] = torch.from_numpy(table).cuda()
    s["slots"] = torch.from_numpy(np.concatenate(slots).astype(np.int32)).cuda()
    s["err"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    s["ws_bytes"] = 0
    if case["entry"] == "workspace":
        s["ws_bytes"] = ppas.ppas_attention_workspace_size(s["q_lens"], s["ctx_lens"], hq, hk)
        s["ws"] = torch.empty(max(s["ws_bytes"], 256), dtype=torch.uint8, device="cuda")
    s["layers"] = []
    for n in range(case["layers"]):
        z = (seed * 64 + n) * 8
        s["layers"].append({
            "q": _normal((s["tokens"], hq, DIM), z + 1) * case["gain"],
            "k_new": _normal((s["tokens"], hk, DIM), z + 2), "v_new": _normal((s["tokens"], hk, DIM), z + 3),
            "k": _normal((s["blocks"], hk, PAGE, DIM), z + 4), "v": _normal((s["blocks"], hk, PAGE, DIM), z + 5),
            "out": torch.empty((s["tokens"], hq, DIM), dtype=torch.float32 if case["fp32"] else torch.bfloat16,
                               device="cuda")})
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    case = s["case"]
    if case["kind"] == "gateup":
        ppas.ppas_gateup_swiglu(s["x"], s["packed"], s["y"], case["tokens"], case["hidden"], case["inter"], s["err"])
        return s["y"]
    hq, hk, scale = case["hq"], case["hk"], DIM ** -0.5
    for y in s["layers"]:
        ppas.ppas_kv_append(y["k_new"], y["v_new"], s["slots"], s["tokens"], y["k"], y["v"], s["blocks"], hk, DIM,
                            s["err"])
        if case["entry"] == "workspace":
            ppas.ppas_attention_step(y["q"], y["k"], y["v"], s["blocks"], s["table"], s["width"], s["q_lens"],
                                     s["ctx_lens"], hq, hk, DIM, scale, y["out"], case["fp32"], s["ws"],
                                     s["ws_bytes"], s["err"])
        else:
            ppas.ppas_attention_step_noalloc(y["q"], y["k"], y["v"], s["blocks"], s["table"], s["width"],
                                             s["q_lens"], s["ctx_lens"], hq, hk, DIM, scale, y["out"], case["fp32"],
                                             s["err"])
    return {"out": [y["out"] for y in s["layers"]], "k": [y["k"] for y in s["layers"]],
            "v": [y["v"] for y in s["layers"]], "err": s["err"]}


def work(case):
    if case["kind"] == "gateup":
        t, h, i = case["tokens"], case["hidden"], case["inter"]
        return {"bytes": 2 * (t * h + 2 * i * h + t * i), "flops": 2 * t * h * 2 * i}
    q, ctx = _lens(case)
    hq, hk = case["hq"], case["hk"]
    pairs = sum(a * (c - a) + a * (a + 1) // 2 for a, c in zip(q, ctx))
    # K and V of every context read, the new tokens' read and written, Q read, the output written
    kv = (sum(ctx) + 2 * sum(q)) * hk * DIM * 4
    return {"bytes": case["layers"] * (kv + sum(q) * hq * DIM * (6 if case["fp32"] else 4)),
            "flops": case["layers"] * 4 * DIM * hq * pairs}


def tolerance(case):
    # the weights of the weighted sum are rounded to bf16 in either kind of
    # row, against maxima that may differ by implementation, and most outputs
    # are bf16
    if case["kind"] == "gateup":
        return {"rel": 0.004, "max": 0.02}
    return {"rel": 0.01, "max": 0.05}


# ------------------------------------------------------------------ the same in 64 bits
def _softmax_rows(q, k, v, first, scale):
    """softmax(scale q k^T) v of query rows at positions first, first + 1, ...
    over keys 0 .. k.shape[0] - 1, causal; float64."""
    w = (q @ k.T) * scale
    pos = torch.arange(first, first + q.shape[0], device=q.device)
    w.masked_fill_(torch.arange(k.shape[0], device=q.device)[None, :] > pos[:, None], float("-inf"))
    return torch.softmax(w, dim=-1) @ v


def exact(case, seed):
    s = prepare(case, seed)
    if case["kind"] == "gateup":
        i = case["inter"]
        w = s["w"].double()
        out = []
        for a in range(0, case["tokens"], 2048):
            p = s["x"][a:a + 2048].double() @ w.T
            out.append(p[:, :i] * torch.sigmoid(p[:, :i]) * p[:, i:])
        return torch.cat(out)
    group, scale = case["hq"] // case["hk"], DIM ** -0.5
    got = {"out": [], "k": [], "v": [], "err": None}
    slots = s["slots"].long()
    for y in s["layers"]:
        for n in ("k", "v"):
            y[n][slots // PAGE, :, slots % PAGE] = y[n + "_new"]
            got[n].append(y[n].double())
        out = torch.empty(y["out"].shape, dtype=torch.float64, device="cuda")
        at = 0
        for r, (nq, c) in enumerate(zip(s["q_lens"].tolist(), s["ctx_lens"].tolist())):
            pages = torch.from_numpy(s["table_host"][r, :-(-c // PAGE)]).cuda().long()
            for kvh in range(case["hk"]):
                k = y["k"][pages, kvh].reshape(-1, DIM)[:c].double()
                v = y["v"][pages, kvh].reshape(-1, DIM)[:c].double()
                heads = range(kvh * group, (kvh + 1) * group)
                if nq == 1:
                    w = torch.softmax((y["q"][at, heads.start:heads.stop].double() @ k.T) * scale, dim=-1)
                    out[at, heads.start:heads.stop] = w @ v
                    continue
                for h in heads:
                    for a in range(0, nq, 2048):
                        b = min(nq, a + 2048)
                        last = c - nq + b
                        out[at + a:at + b, h] = _softmax_rows(y["q"][at + a:at + b, h].double(), k[:last], v[:last],
                                                              c - nq + a, scale)
            at += nq
        got["out"].append(out)
    return got
