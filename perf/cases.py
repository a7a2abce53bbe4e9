"""The work that a user of the library has it do, as cases to be timed and compared.

Every case is one call of a public entry point of ``dck`` (the C ABI's binding)
on a layer's caches, factors and workspace, held the way a serving loop holds
them.  Kinds:

  step     dck_decode_step: the batch's new tokens appended, then one query
           per sequence over the caches (returns the output and both caches)
  attend   dck_decode_attention: the query half of a step alone
  append   dck_latent_append: new tokens' latents into given cache rows
  prefill  dck_prefill_attention: a prompt, or the next chunk of one, attending
           causally to its prefix

Sequence lengths are ``lo == hi`` (all alike) or ragged, drawn log-uniformly
from [lo, hi] with ``lens_seed``.  ``cap`` > 0 gives every sequence that many
rows of a pooled cache (the rows behind its tokens hold other data); 0 packs
the sequences back to back.
"""

import math
import random

import torch

from paper_2607_24331_gb300 import dck

# The repository's layer shapes: group sizes and ranks of the keys, value rank.
LAYERS = {
    # fp32 MHA layer
    "mha8-f32": dict(hidden=512, hq=8, hkv=8, d=64, sizes=(3, 5), ranks=(48, 96), rv=160, theta=1e4, f32=True),
    # 32-head MHA layer, uneven key groups
    "mha32": dict(hidden=4096, hq=32, hkv=32, d=128, sizes=(2, 3, 3, 4, 4, 5, 5, 6),
                  ranks=(64, 96, 96, 128, 128, 160, 160, 192), rv=1024, theta=1e4, f32=False),
    # the same with fixed groups of four
    "mha32-fixed": dict(hidden=4096, hq=32, hkv=32, d=128, sizes=(4,) * 8, ranks=(128,) * 8, rv=1024, theta=1e4,
                        f32=False),
    # GQA layers, 32 query and 8 KV heads
    "gqa8": dict(hidden=4096, hq=32, hkv=8, d=128, sizes=(1, 1, 2, 2, 2), ranks=(96, 96, 160, 192, 224), rv=512,
                 theta=1e6, f32=False),
    "gqa8-long": dict(hidden=4096, hq=32, hkv=8, d=128, sizes=(2, 3, 3), ranks=(192, 256, 256), rv=384, theta=5e5,
                      f32=False),
}


def _heads(L):
    """KV heads in group order: a fixed permutation, since head grouping leaves no contiguous order."""
    return [(5 * i + 3) % L["hkv"] for i in range(L["hkv"])]


def _case(name, kind, layer, batch, lo, hi, q_lo=0, q_hi=0, cap=0, tokens=0, lens_seed=1):
    c = dict(kind=kind, layer=layer, batch=batch, lo=lo, hi=hi, q_lo=q_lo, q_hi=q_hi, cap=cap, tokens=tokens,
             lens_seed=lens_seed)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one decode step of the fp32 layer, one user
        _case("step-f32-b1-512", "step", "mha8-f32", 1, 512, 512),
        # one decode step for one user in a short conversation: latency
        _case("step-mha-b1-777", "step", "mha32", 1, 777, 777),
        # the ordinary serving batch (the benchmark's default workload)
        _case("step-mha-b16-4096", "step", "mha32", 16, 4096, 4096),
        # a continuous batch: every sequence of another length, in a pooled cache
        _case("step-mha-b32-ragged", "step", "mha32", 32, 1024, 16384, cap=16384),
        # a GQA layer's batch at its context limit
        _case("step-gqa-b8-32768", "step", "gqa8", 8, 32768, 32768),
        # the longest contexts: two documents of 128k tokens
        _case("attend-gqa-b2-131072", "attend", "gqa8-long", 2, 131072, 131072),
        # latents of a small set of tokens (speculative or draft tokens of a batch), scattered rows
        _case("append-mha-100", "append", "mha32", 1, 0, 0, tokens=100),
        # latents of a long prompt pair
        _case("append-gqa-16384", "append", "gqa8-long", 1, 0, 0, tokens=16384),
        # a few short prompts of odd lengths
        _case("prefill-mha-b8-short", "prefill", "mha32", 8, 33, 300, q_lo=33, q_hi=300),
        # two whole prompts
        _case("prefill-mha-b2-4096", "prefill", "mha32", 2, 4096, 4096, q_lo=4096, q_hi=4096),
        # one long whole prompt on a GQA layer
        _case("prefill-gqa-b1-8192", "prefill", "gqa8-long", 1, 8192, 8192, q_lo=8192, q_hi=8192),
        # chunked prefill: the next chunk of several prompts, in a pooled cache
        _case("prefill-gqa-b4-chunk", "prefill", "gqa8", 4, 2000, 7000, q_lo=300, q_hi=512, cap=16384),
    ]


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


MAX_PREFILL_PAIRS = 8192 * 8192  # queries x keys of one KV group's heads, summed over the batch
MAX_ROWS = 262144                # cache rows of a decode call


def draw(rng):
    kind = rng.choice(("step", "step", "step", "attend", "append", "prefill", "prefill", "f32"))
    seed = rng.randrange(1 << 20)
    layer = rng.choice(("mha32", "mha32-fixed", "gqa8", "gqa8-long"))
    if kind == "f32":
        return _case(None, "step", "mha8-f32", rng.randint(1, 8), 1, _logint(rng, 16, 4096), lens_seed=seed)
    if kind == "append":
        return _case(None, "append", layer, 1, 0, 0, tokens=_logint(rng, 1, 16384), lens_seed=seed)
    if kind == "prefill":
        while True:
            b, hi = _logint(rng, 1, 16), _logint(rng, 32, 8192)
            lo = rng.choice((hi, max(1, hi // 4)))
            q_hi = rng.choice((hi, _logint(rng, 1, min(hi, 1024))))
            if b * q_hi * hi <= MAX_PREFILL_PAIRS // 2:
                q_lo = min(lo, max(1, q_hi // 2)) if q_hi < hi else lo
                return _case(None, "prefill", layer, b, lo, hi, q_lo=q_lo, q_hi=q_hi,
                             cap=rng.choice((0, 4 * hi)) if b * hi <= 16384 else 0, lens_seed=seed)
    while True:
        b, hi = _logint(rng, 1, 64), _logint(rng, 64, 131072)
        if b * hi <= (MAX_ROWS if layer.startswith("gqa") else MAX_ROWS // 2):
            lo = rng.choice((hi, max(1, hi // 16)))
            return _case(None, kind, layer, b, lo, hi, cap=rng.choice((0, hi)) if lo < hi else 0, lens_seed=seed)


def _lens(case):
    """(lengths, query lengths) of the batch."""
    rng = random.Random(case["lens_seed"])
    lens = [_logint(rng, case["lo"], case["hi"]) for _ in range(case["batch"])]
    q = [0] * len(lens)
    if case["kind"] == "prefill":
        whole = case["q_lo"] == case["lo"] and case["q_hi"] == case["hi"]
        q = [n if whole else min(n, _logint(rng, case["q_lo"], case["q_hi"])) for n in lens]
    return lens, q


def _inputs(case, seed):
    """The call's tensors, in plain torch: unit-variance latents and hidden states, factors scaled so that
    keys and values have unit variance, queries of twice that (scores of standard deviation 2)."""
    L = LAYERS[case["layer"]]
    dt = torch.float32 if L["f32"] else torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(shape, std=1.0):
        return torch.randn(shape, generator=gen, device="cuda", dtype=dt).mul_(std)

    rk, rv, D = sum(L["ranks"]), L["rv"], L["hidden"]
    t = {}
    if case["kind"] == "append":
        n = case["tokens"]
        t["n_rows"] = n + n // 2 + 8
        t["rows"] = torch.randperm(t["n_rows"], generator=gen, device="cuda")[:n].contiguous()
        if n > 1024:  # a prompt's rows lie one after the other
            t["rows"] = t["rows"].sort().values
        t["kcache"] = torch.zeros((t["n_rows"], rk), dtype=dt, device="cuda")
        t["vcache"] = torch.zeros((t["n_rows"], rv), dtype=dt, device="cuda")
    else:
        lens, q_lens = _lens(case)
        cap = max(case["cap"], max(lens)) if case["cap"] else 0
        starts, at = [], 0
        for n in lens:
            starts.append(at)
            at += cap or n
        t["n_rows"] = at
        t["seq_start"] = torch.tensor(starts, dtype=torch.int64, device="cuda")
        t["seq_len"] = torch.tensor(lens, dtype=torch.int32, device="cuda")
        t["kcache"] = normal((at, rk))
        t["vcache"] = normal((at, rv))
        t["B_k"] = torch.cat([normal((r * n * L["d"],), 1 / math.sqrt(r)) for n, r in zip(L["sizes"], L["ranks"])])
        t["B_v"] = normal((rv, L["hkv"] * L["d"]), 1 / math.sqrt(rv))
        if case["kind"] == "prefill":
            t["q_len"] = torch.tensor(q_lens, dtype=torch.int32, device="cuda")
            t["q"] = normal((case["batch"], max(q_lens), L["hq"], L["d"]), 2.0)
        else:
            t["q"] = normal((case["batch"], L["hq"], L["d"]), 2.0)
            t["rows"] = t["seq_start"] + t["seq_len"] - 1
        t["out"] = torch.zeros_like(t["q"])
    if case["kind"] in ("append", "step"):
        t["x"] = normal((case["tokens"] if case["kind"] == "append" else case["batch"], D))
        t["A_k"] = normal((D, rk), 1 / math.sqrt(D))
        t["A_v"] = normal((D, rv), 1 / math.sqrt(D))
    return t


def prepare(case, seed):
    L = LAYERS[case["layer"]]
    t = _inputs(case, seed)
    heads, groups = _heads(L), []
    for n in L["sizes"]:
        groups.append(heads[:n])
        heads = heads[n:]
    layer = dck.Layer(L["hidden"], L["hq"], L["hkv"], L["d"], groups, L["ranks"], L["rv"], "f32" if L["f32"] else "bf16")
    b = case["batch"]
    size = {"step": lambda: dck.dck_decode_step_workspace_size(layer, b, t["n_rows"]),
            "attend": lambda: dck.dck_decode_workspace_size(layer, b, t["n_rows"]),
            "append": lambda: dck.dck_latent_append_workspace_size(layer, case["tokens"]),
            "prefill": lambda: dck.dck_prefill_workspace_size(layer, t["n_rows"])}[case["kind"]]()
    ws = torch.empty(max(size, 256), dtype=torch.uint8, device="cuda")
    lens = _lens(case)[0] if case["kind"] == "prefill" else [0]
    return {"kind": case["kind"], "layer": layer, "batch": b, "theta": L["theta"], "ws": ws, "ws_bytes": size,
            "max_len": max(lens), **t}


def run(s):
    kind = s["kind"]
    if kind == "step":
        dck.check(dck.dck_decode_step(s["layer"], s["x"], s["A_k"], s["A_v"], s["rows"], s["q"], s["kcache"],
                                      s["vcache"], s["n_rows"], s["B_k"], s["B_v"], s["seq_start"], s["seq_len"],
                                      s["batch"], s["theta"], s["out"], s["ws"], s["ws_bytes"]), "dck_decode_step")
        return {"out": s["out"], "kcache": s["kcache"], "vcache": s["vcache"]}
    if kind == "attend":
        dck.check(dck.dck_decode_attention(s["layer"], s["q"], s["kcache"], s["vcache"], s["n_rows"], s["B_k"],
                                           s["B_v"], s["seq_start"], s["seq_len"], s["batch"], s["theta"], s["out"],
                                           s["ws"], s["ws_bytes"]), "dck_decode_attention")
        return {"out": s["out"]}
    if kind == "append":
        dck.check(dck.dck_latent_append(s["layer"], s["x"], s["x"].shape[0], s["A_k"], s["A_v"], s["rows"],
                                        s["kcache"], s["vcache"], s["n_rows"], s["ws"], s["ws_bytes"]),
                  "dck_latent_append")
        return {"kcache": s["kcache"], "vcache": s["vcache"]}
    dck.check(dck.dck_prefill_attention(s["layer"], s["q"], s["q_len"], s["q"].shape[1], s["kcache"], s["vcache"],
                                        s["n_rows"], s["B_k"], s["B_v"], s["seq_start"], s["seq_len"], s["batch"],
                                        s["max_len"], s["theta"], s["out"], s["ws"], s["ws_bytes"]),
              "dck_prefill_attention")
    return {"out": s["out"]}


def work(case):
    """Caches' rows in use, factors, hidden states and queries read once, outputs written once; the
    products of the method (append, key and value reconstruction or absorption, scores, P V)."""
    L = LAYERS[case["layer"]]
    el = 4 if L["f32"] else 2
    rk, rv, D, hq, hkv, d = sum(L["ranks"]), L["rv"], L["hidden"], L["hq"], L["hkv"], L["d"]
    rec = sum(r * n for r, n in zip(L["ranks"], L["sizes"])) * d  # multiply-adds of one token's keys
    if case["kind"] == "append":
        n = case["tokens"]
        return {"bytes": el * (n * (D + rk + rv) + D * (rk + rv)) + 8 * n, "flops": 2 * n * D * (rk + rv)}
    lens, q_lens = _lens(case)
    rows, b = sum(lens), case["batch"]
    factors = rec + rv * hkv * d
    if case["kind"] == "prefill":
        pairs = sum(q * (n - q) + q * (q + 1) // 2 for n, q in zip(lens, q_lens))
        return {"bytes": el * (rows * (rk + rv) + factors + 2 * sum(q_lens) * hq * d) + 16 * b,
                "flops": 2 * rows * (rec + rv * hkv * d) + 4 * pairs * hq * d}
    w = {"bytes": el * (rows * (rk + rv) + factors + 2 * b * hq * d) + 12 * b,
         "flops": 2 * rows * (rec + hq * d + hq * rv) + 2 * b * hq * rv * d}
    if case["kind"] == "step":
        w["bytes"] += el * (D * (rk + rv) + b * (D + rk + rv)) + 8 * b
        w["flops"] += 2 * b * D * (rk + rv)
    return w


def tolerance(case):
    if LAYERS[case["layer"]]["f32"]:
        return {"rel": 1e-5}
    if case["kind"] == "append":
        return {"rel": 2e-3}  # one bf16 rounding of an fp32 sum: another order of the sum moves a few of them by an ulp
    # four times the error against 64 bits seen in the output (probabilities, key factors or keys and queries in
    # bf16): 3.5e-3 where the query is folded into the factors, 5e-3 to 6.6e-3 where keys are rotated and rounded
    return {"rel": 1.4e-2 if case["kind"] != "prefill" and case["layer"].startswith("mha32") else 2e-2}


def _rope(x, pos, theta):
    """Rotate-half RoPE of x [..., d] at positions pos (broadcast against x's leading axes)."""
    d = x.shape[-1]
    w = torch.pow(torch.tensor(float(torch.tensor(theta, dtype=torch.float32)), dtype=torch.float64, device=x.device),
                  -2.0 * torch.arange(d // 2, dtype=torch.float64, device=x.device) / d)
    a = pos.to(torch.float64).unsqueeze(-1) * w
    c, s = torch.cos(a), torch.sin(a)
    x1, x2 = x[..., : d // 2], x[..., d // 2:]
    return torch.cat([x1 * c - x2 * s, x1 * s + x2 * c], -1)


def exact(case, seed):
    L = LAYERS[case["layer"]]
    t = _inputs(case, seed)
    hq, hkv, d, theta = L["hq"], L["hkv"], L["d"], L["theta"]
    f64 = torch.float64
    dt = t["kcache"].dtype
    got = {}
    if case["kind"] in ("append", "step"):
        x = t["x"].to(f64)
        ck, cv = x @ t["A_k"].to(f64), x @ t["A_v"].to(f64)
        kc, vc = t["kcache"].to(f64), t["vcache"].to(f64)
        kc[t["rows"]], vc[t["rows"]] = ck, cv
        got["kcache"], got["vcache"] = kc, vc
        if case["kind"] == "append":
            return got
        t["kcache"][t["rows"]], t["vcache"][t["rows"]] = ck.to(dt), cv.to(dt)  # caches hold their storage type
    lens, q_lens = _lens(case)
    qpg = hq // hkv
    heads = _heads(L)
    B_v = t["B_v"].to(f64).view(L["rv"], hkv, d)
    out = torch.zeros(t["out"].shape, dtype=f64, device="cuda")
    at = [int(v) for v in t["seq_start"].cpu()]
    for b, n in enumerate(lens):
        pos = torch.arange(n, device="cuda")
        v = t["vcache"][at[b]: at[b] + n].to(f64)
        r0 = b0 = h0 = 0
        for size, r in zip(L["sizes"], L["ranks"]):
            B_g = t["B_k"][b0: b0 + r * size * d].to(f64).view(r, size, d)
            c = t["kcache"][at[b]: at[b] + n, r0: r0 + r].to(f64)
            for slot in range(size):
                h = heads[h0 + slot]
                k = _rope(c @ B_g[:, slot], pos, theta)
                js = slice(h * qpg, (h + 1) * qpg)
                if case["kind"] == "prefill":
                    vh = v @ B_v[:, h]
                    for i0 in range(0, q_lens[b], 2048):
                        i1 = min(q_lens[b], i0 + 2048)
                        p = n - q_lens[b] + torch.arange(i0, i1, device="cuda")
                        q = _rope(t["q"][b, i0:i1, js].to(f64), p.unsqueeze(1), theta)
                        s = torch.einsum("qjd,td->jqt", q, k) / math.sqrt(d)
                        s.masked_fill_(pos > p.unsqueeze(1), -math.inf)
                        out[b, i0:i1, js] = torch.einsum("jqt,td->qjd", torch.softmax(s, -1), vh)
                else:
                    q = _rope(t["q"][b, js].to(f64), torch.full((1,), n - 1, device="cuda"), theta)
                    u = torch.softmax(q @ k.T / math.sqrt(d), -1) @ v
                    out[b, js] = u @ B_v[:, h]
            r0, b0, h0 = r0 + r, b0 + r * size * d, h0 + size
    got["out"] = out
    return got
