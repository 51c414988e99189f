"""Performance cases of libgc: what a serving program has it do, layer by layer.

A case is one pass of one of these paths through the C ABI's Python binding:

* ``step``       restore of the cached pages from a device image, append of
                 the new tokens' K/V, prefill attention (one layer)
* ``host-step``  the same with the cached pages in pinned host memory, staged
                 through device memory
* ``decode``     append of one token per request, paged decode attention
* ``q8-prefill`` append and prefill attention, full cached pages read from the
                 8-bit cache tier
* ``q8-decode``  the same for decode
* ``tier``       cached pages of several layers saved to the cache tier in
                 bf16 and in 8 bits, and restored from the 8-bit image

Fields: ``B`` requests; ``hq`` / ``hkv`` heads of size ``d``; pages of ``ps``
tokens; ``L`` layers of the pool (attention runs on the last).  Lengths come
from ``lens`` (their seed) alone: ``spread`` "fixed" gives every request
``prefix`` cached and ``new`` new tokens, "uniform" draws both up to those
bounds (from an eighth of ``prefix`` and a quarter of ``new`` on), "lognormal"
takes them as medians of multi-turn traffic, where a request misses the cache
(its whole context is then new) with probability ``1 - hit``.
"""
import math

import numpy as np
import torch

from paper_2505_23970_gb300 import binding as gcb

_BF16 = torch.bfloat16


def _case(name, kind, B, hq, hkv, d, ps, prefix, new, spread="fixed", L=1, hit=1.0, lens=0):
    c = dict(kind=kind, B=B, hq=hq, hkv=hkv, d=d, ps=ps, prefix=prefix, new=new, spread=spread,
             L=L, hit=hit, lens=lens)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one short request of a small GQA 4:1 model with
        # head size 64; latency and launches are all there is
        _case("tiny-step-d64", "step", 1, 4, 1, 64, 16, 256, 64),
        # one interactive chat turn of a Llama-3-8B-shaped layer: a short
        # question after a cached conversation that is still in host memory
        _case("chat-turn-8b", "host-step", 1, 32, 8, 128, 16, 1873, 43),
        # continuous batching on a Llama-3-8B-shaped layer, ragged lengths
        _case("layer-8b", "step", 16, 32, 8, 128, 16, 4096, 512, "uniform"),
        # a batch of long cached prefixes on a Llama-3-70B-shaped layer
        _case("layer-70b", "step", 8, 64, 8, 128, 16, 8192, 1024),
        # multi-turn traffic on the 70B-shaped layer, half of the requests
        # missing the cache: short and long, reused and from scratch
        _case("conversation-mix", "step", 64, 64, 8, 128, 16, 2048, 200, "lognormal", hit=0.5),
        # questions on two long documents, 131072 cached tokens each: the
        # largest call
        _case("long-document", "step", 2, 64, 8, 128, 64, 131072, 2048),
        # ragged batch of a model with head size 64
        _case("layer-d64", "step", 12, 32, 8, 64, 16, 3001, 701, "uniform"),
        # generation on the 70B-shaped layer, eight requests of equal context
        _case("decode-70b", "decode", 8, 64, 8, 128, 16, 9215, 1),
        # generation with a few short contexts, head size 64
        _case("decode-d64", "decode", 5, 32, 8, 64, 16, 1900, 1, "uniform"),
        # the cached prefixes stay in the 8-bit tier: prefill over them ...
        _case("q8-prefill-70b", "q8-prefill", 4, 64, 8, 128, 16, 8000, 900, "uniform"),
        # ... and generation with many contexts of multi-turn length
        _case("q8-decode-mix", "q8-decode", 64, 64, 8, 128, 16, 2248, 1, "lognormal"),
        # a finished request's pages leave for the cache tier, in either
        # precision, and another's come back from 8 bits
        _case("tier-16-layers", "tier", 3, 64, 8, 128, 16, 3456, 0, "uniform", L=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "host-step", "decode", "decode", "q8-prefill",
                       "q8-decode", "tier"])
    d = rng.choice([64, 128, 128])
    hkv = rng.choice([1, 2, 4, 8, 8])
    hq = hkv * rng.choice([1, 4, 8, 8, 16])
    ps = rng.choice([16, 16, 32, 64, 128])
    spread = rng.choice(["fixed", "uniform", "lognormal"])
    hit = rng.choice([1.0, 1.0, 0.5]) if kind == "step" else 1.0
    lens = rng.randrange(1 << 20)
    if kind == "tier":
        return _case("", kind, _log(rng, 1, 16), hq, hkv, d, ps, _log(rng, 100, 4000), 0, spread,
                     rng.choice([1, 2, 5, 16]), 1.0, lens)
    B = _log(rng, 1, 16 if kind == "host-step" else 128)
    prefix = _log(rng, 32, 4096 if kind == "host-step" else 32768)
    new = 1 if "decode" in kind else _log(rng, 1, 2048)
    c = _case("", kind, B, hq, hkv, d, ps, prefix, new, spread, 1, hit, lens)
    # no dearer than the largest listed case
    while c["B"] > 1 and (work(c)["flops"] > 6e12 or work(c)["bytes"] > 1.5e9):
        c["B"] //= 2
    return c


# ---------------------------------------------------------------- lengths
def _lens(c):
    """(cached, new) tokens of each request."""
    B, P, n = c["B"], c["prefix"], c["new"]
    rng = np.random.default_rng([c["lens"], 1])
    if c["spread"] == "fixed":
        return np.full(B, P, np.int64), np.full(B, n, np.int64)
    if c["spread"] == "uniform":
        return (rng.integers(max(0, P // 8), P, size=B, endpoint=True),
                rng.integers(max(min(n, 1), n // 4), n, size=B, endpoint=True))
    p = np.clip(np.rint(rng.lognormal(math.log(P), 1.0, size=B)), 0, 16 * P).astype(np.int64)
    s = np.clip(np.rint(rng.lognormal(math.log(max(n, 1)), 0.8, size=B)), max(1, n // 12),
                20 * max(n, 1)).astype(np.int64)
    if n <= 1:
        s = np.full(B, n, np.int64)
    hit = np.random.default_rng([c["lens"], 2]).random(B) < c["hit"]
    return np.where(hit, p, 0), np.where(hit, s, p + s)


def _page_counts(c):
    """Per request: pages of the whole sequence, pages of the cached prefix,
    and full cached pages (those an 8-bit image holds)."""
    P, n = _lens(c)
    ps = c["ps"]
    return -(-(P + n) // ps), -(-P // ps), P // ps


def _chunk(c):
    """bf16 bytes of one page of one layer and plane."""
    return c["hkv"] * c["ps"] * c["d"] * 2


def _q8_header(c):
    return (c["hkv"] * 4 + 15) // 16 * 16


# ----------------------------------------------------------------- inputs
def _randn(gen, shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=_BF16)


def _quantise(x):
    """8-bit image [n][L][2][chunk] of bf16 pages [n][L][2][hkv][ps][d]."""
    n, L, _, hkv, ps, d = x.shape
    f = x.float().view(n, L, 2, hkv, ps * d)
    amax = f.abs().amax(-1, keepdim=True)
    codes = torch.round(f * (127.0 / amax)).clamp(-127, 127).to(torch.int8)
    head = torch.zeros((n, L, 2, (hkv * 4 + 15) // 16 * 4), dtype=torch.float32, device=x.device)
    head[..., :hkv] = (amax / 127.0).squeeze(-1)
    return torch.cat([head.view(torch.uint8).view(n, L, 2, -1),
                      codes.view(torch.uint8).view(n, L, 2, -1)], -1).contiguous()


def _dequantise(c, image):
    n = image.shape[0]
    h = _q8_header(c)
    scale = image[..., :h].contiguous().view(torch.float32)[..., :c["hkv"]]
    codes = image[..., h:].contiguous().view(torch.int8).view(n, c["L"], 2, c["hkv"], c["ps"], c["d"])
    return (codes.float() * scale[..., None, None]).to(_BF16)


def _i32(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()


def _inputs(c, seed):
    """The inputs of a case as plain tensors.  ``pool``: the pool's contents
    before the pass (other requests' pages, and this batch's cached pages where
    the pass does not restore them)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    P, n = _lens(c)
    total, cached, full = _page_counts(c)
    pages = max(1, math.ceil(1.25 * int(total.sum())))
    perm = np.random.default_rng([int(seed) & 0x7FFFFFFF, 3]).permutation(pages)
    table = np.full((c["B"], max(1, int(total.max()))), -1, np.int64)
    at = 0
    for b, k in enumerate(total):
        table[b, :k] = perm[at:at + k]
        at += int(k)
    hkv, ps, d, L = c["hkv"], c["ps"], c["d"], c["L"]
    x = dict(P=P, n=n, table=table, pages=pages,
             pool=_randn(gen, (L, 2, pages, hkv, ps, d)))
    kind = c["kind"]
    if kind != "tier":
        T = int(n.sum())
        x["q"], x["k"] = _randn(gen, (T, c["hq"], d)), _randn(gen, (T, hkv, d))
        x["v"] = _randn(gen, (T, hkv, d))
        x["cu"] = np.concatenate([[0], np.cumsum(n)])
    count = full if kind.startswith("q8") else cached
    x["ids"] = np.concatenate([table[b, :k] for b, k in enumerate(count)])
    blocks = x["ids"].size
    if kind in ("step", "host-step"):
        x["image"] = _randn(gen, (blocks, L, 2, hkv, ps, d))
    elif kind != "decode":
        x["image"] = _quantise(_randn(gen, (blocks, L, 2, hkv, ps, d)))
        q8 = np.full(table.shape, -1, np.int64)
        at = 0
        for b, k in enumerate(full):
            q8[b, :k] = np.arange(at, at + k)
            at += int(k)
        x["q8"] = q8
    return x


def prepare(case, seed):
    c = dict(case)
    x = _inputs(c, seed)
    kind, blocks = c["kind"], int(x["ids"].size)
    pool = gcb.KVPool.create(c["L"], c["hkv"], c["d"], c["ps"], x["pages"])
    pool.planes().copy_(x["pool"])
    s = dict(kind=kind, pool=pool, handle=pool.handle, planes=pool.planes(), L=c["L"],
             layer=c["L"] - 1, blocks=blocks, B=c["B"], hq=c["hq"], scale=c["d"] ** -0.5,
             width=x["table"].shape[1], table=_i32(x["table"]), ids=_i32(x["ids"]),
             stream=torch.cuda.current_stream())
    if kind == "tier":
        s["q8_in"] = x["image"]
        s["bf16_out"] = torch.zeros((blocks, c["L"], 2, c["hkv"], c["ps"], c["d"]), dtype=_BF16,
                                    device="cuda")
        s["q8_out"] = torch.zeros_like(x["image"])
        return s
    s["T"] = int(x["n"].sum())
    s["q"], s["k"], s["v"] = x["q"], x["k"], x["v"]
    s["out"] = torch.zeros_like(x["q"])
    s["prefix"], s["new"], s["cu"] = _i32(x["P"]), _i32(x["n"]), _i32(x["cu"])
    if kind == "step":
        s["image"] = x["image"]
    elif kind == "host-step":
        s["image"] = torch.empty(x["image"].shape, dtype=_BF16, pin_memory=True)
        s["image"].copy_(x["image"])
        s["staging"] = torch.empty_like(x["image"])
    if kind.startswith("q8"):
        s["image"], s["q8"] = x["image"], _i32(x["q8"])
    if kind.endswith("decode"):
        s["seq"] = _i32(x["P"] + x["n"])
        s["need"] = gcb.gc_paged_decode_workspace_bytes(s["handle"], s["B"], s["width"], s["hq"])
        s["work"] = torch.empty(max(16, s["need"]), dtype=torch.uint8, device="cuda")
    return s


# ------------------------------------------------------------------- pass
def run(s):
    kind, h, st = s["kind"], s["handle"], s["stream"]
    if kind == "tier":
        gcb.gc_kv_save(h, s["bf16_out"], s["ids"], s["blocks"], st, None, gcb.GC_SAVE_DST_DEVICE)
        gcb.gc_kv_save_q8(h, s["q8_out"], s["ids"], s["blocks"], 0, s["L"], st, None,
                          gcb.GC_SAVE_DST_DEVICE)
        gcb.gc_kv_restore_q8(h, s["q8_in"], s["ids"], s["blocks"], 0, s["L"], st, None,
                             gcb.GC_RESTORE_SRC_DEVICE)
        return {"bf16": s["bf16_out"], "q8": s["q8_out"], "kv": s["planes"]}
    if kind == "step":
        gcb.gc_kv_restore(h, s["image"], s["ids"], s["blocks"], st, None, gcb.GC_RESTORE_SRC_DEVICE)
    elif kind == "host-step":
        gcb.gc_kv_restore(h, s["image"], s["ids"], s["blocks"], st, s["staging"], 0)
    gcb.gc_kv_append(h, s["k"], s["v"], s["table"], s["prefix"], st, s["layer"], s["cu"], s["B"],
                     s["width"], s["T"])
    if kind == "decode":
        gcb.gc_paged_decode_attn(s["q"], h, s["table"], s["seq"], s["out"], st, s["layer"], s["B"],
                                 s["width"], s["hq"], s["scale"], s["work"], s["need"])
    elif kind == "q8-decode":
        gcb.gc_paged_decode_attn_q8(s["q"], h, s["table"], s["seq"], s["out"], st, s["layer"],
                                    s["B"], s["width"], s["hq"], s["scale"], s["work"], s["need"],
                                    s["image"], s["q8"], s["blocks"], 0)
    elif kind == "q8-prefill":
        gcb.gc_prefix_prefill_attn_q8(s["q"], h, s["table"], s["prefix"], s["new"], s["out"], st,
                                      s["layer"], s["cu"], s["B"], s["width"], s["hq"], s["scale"],
                                      s["T"], s["image"], s["q8"], s["blocks"], 0)
    else:
        gcb.gc_prefix_prefill_attn(s["q"], h, s["table"], s["prefix"], s["new"], s["out"], st,
                                   s["layer"], s["cu"], s["B"], s["width"], s["hq"], s["scale"],
                                   s["T"])
    return {"out": s["out"], "kv": s["planes"]}


def work(c):
    P, n = _lens(c)
    _, cached, full = _page_counts(c)
    kind = c["kind"]
    if kind == "tier":
        # the saves' shared input, both images written, the 8-bit image read,
        # the restored pages written
        b16 = int(cached.sum()) * c["L"] * 2 * _chunk(c)
        b8 = int(cached.sum()) * c["L"] * 2 * (_q8_header(c) + _chunk(c) // 2)
        return {"bytes": 3 * b16 + 2 * b8, "flops": 0}
    row = c["hkv"] * c["d"] * 2 * 2  # one token's K and V
    T = int(n.sum())
    new = 2 * T * row                        # appended: read, written
    qo = 2 * T * c["hq"] * c["d"] * 2        # q read, out written
    flops = 4.0 * c["d"] * c["hq"] * float(np.sum(n * P + n * (n + 1) / 2))
    if kind in ("step", "host-step"):
        kv = int(cached.sum()) * 2 * 2 * _chunk(c)  # the image read, its pages written
    elif kind == "decode":
        kv = int(P.sum()) * row
    else:
        kv = int(full.sum()) * 2 * (_q8_header(c) + _chunk(c) // 2) + int((P - full * c["ps"]).sum()) * row
    return {"bytes": kv + new + qo, "flops": flops}


def tolerance(c):
    # the cache tier is copies and codes decided in 32 bits
    if c["kind"] == "tier":
        return "exact"
    # P and the output are rounded to bf16: about 2.5e-3 off 64 bits, and single
    # values a few times that
    return {"rel": 1e-2, "max": 8e-2}


# -------------------------------------------------------------- 64 bits
def _attention(q, k, v, P, scale):
    """Rows P.. of causal attention: q [n][hq][d], k and v [T][hkv][d]."""
    n, hq, d = q.shape
    T, hkv, _ = k.shape
    G = hq // hkv
    out = torch.empty((n, hq, d), dtype=torch.float64, device=q.device)
    rows = max(1, min(n, int(3e8 / (8 * G * T))))
    keys = torch.arange(T, device=q.device)
    for g in range(hkv):
        kg, vg = k[:, g].double(), v[:, g].double()
        for i in range(0, n, rows):
            m = min(rows, n - i)
            s = (q[i:i + m, g * G:(g + 1) * G].double().reshape(m * G, d) @ kg.T) * scale
            last = P + i + torch.arange(m, device=q.device).repeat_interleave(G)
            s.masked_fill_(keys[None] > last[:, None], -math.inf)
            out[i:i + m, g * G:(g + 1) * G] = (torch.softmax(s, -1) @ vg).view(m, G, d)
    return out


def exact(case, seed):
    c = dict(case)
    if work(c)["flops"] > 5e12:
        return None
    x = _inputs(c, seed)
    pool, kind = x["pool"], c["kind"]
    ids = torch.from_numpy(x["ids"]).cuda()
    if kind == "tier":
        saved = pool[:, :, ids].permute(2, 0, 1, 3, 4, 5).contiguous()
        codes = _quantise(saved)
        pool[:, :, ids] = _dequantise(c, x["image"]).permute(1, 2, 0, 3, 4, 5)
        return {"bf16": saved, "q8": codes, "kv": pool}
    if kind in ("step", "host-step"):
        pool[:, :, ids] = x["image"].permute(1, 2, 0, 3, 4, 5)
    layer = pool[c["L"] - 1]
    table = torch.from_numpy(x["table"]).cuda()
    out = torch.empty(x["q"].shape, dtype=torch.float64, device="cuda")
    q8 = _dequantise(c, x["image"])[:, c["L"] - 1] if kind.startswith("q8") else None
    for b in range(c["B"]):
        P, n, lo = int(x["P"][b]), int(x["n"][b]), int(x["cu"][b])
        if n == 0:
            continue
        pos = torch.arange(P, P + n, device="cuda")
        page, slot = table[b, pos // c["ps"]], pos % c["ps"]
        layer[0, page, :, slot] = x["k"][lo:lo + n]
        layer[1, page, :, slot] = x["v"][lo:lo + n]
        used = table[b, :-(-(P + n) // c["ps"])]
        kv = layer[:, used]
        if q8 is not None:
            src = torch.from_numpy(x["q8"][b]).cuda()
            src = src[src >= 0]
            kv[:, :src.numel()] = q8[src].transpose(0, 1)
        kv = kv.transpose(2, 3).reshape(2, -1, c["hkv"], c["d"])[:, :P + n]
        out[lo:lo + n] = _attention(x["q"][lo:lo + n], kv[0], kv[1], P, c["d"] ** -0.5)
    return {"out": out, "kv": pool}
