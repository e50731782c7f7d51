"""Timed cases of the mixed-format KV cache: what a serving process has the library do, through its public calls.

Kinds of case:
  step     one decode step: Append of a token per request, where `retier` is set Demote of the page that
           leaves each request's Recent window, then decode attention.  One layer goes through the
           single-layer calls, several layers through the calls that take all layers at once.
  scored   decode attention that also reports the page mass, then the update of the page scores
  append   Append of a prefill chunk of several requests
  demote   Demote of many full pages (the ageing of a prefilled context), published into the tables
  promote  Promote of many Stale pages, published into the tables

Shapes are those of mkv_workloads (head_dim 128 and 256, 16-token pages and the paper's long pages, both
record formats, first-tokens Anchor span and Recent window in FP8, the rest Stale).  Every pass leaves the
state such that the next pass does the same work again.
"""
import math

import numpy as np
import torch

import paper_2608_23834_b200 as M

DEVICE = "cuda:0"
STAGE_TOKENS = 65536            # tokens of one fill chunk
# tokens x layers x KV heads x head_dim that a drawn case may hold; the largest listed one holds 1.8 times as many
LARGEST = 32 * 32768 * 8 * 128


def _step(name, layers, batch, ctx_min, ctx_max, d, hkv, group, fmt, anchor, recent, spans=0, page=16, retier=False,
          kind="step"):
    return {"name": name, "kind": kind, "layers": layers, "batch": batch, "ctx_min": ctx_min, "ctx_max": ctx_max,
            "head_dim": d, "kv_heads": hkv, "group": group, "format": fmt, "anchor": anchor, "recent": recent,
            "spans": spans, "page": page, "retier": retier}


def _convert(name, kind, pages, d, hkv, fmt, page=16):
    return {"name": name, "kind": kind, "pages": pages, "head_dim": d, "kv_heads": hkv, "format": fmt, "page": page}


def listed():
    return [
        # one short request, one layer: nothing but launches and latency
        _step("decode_tiny", 1, 1, 4096, 4096, 128, 1, 8, 1, 64, 256),
        # start of a few conversations on a 16-layer model: short ragged contexts, all layers in one call
        _step("decode_short_16l", 16, 4, 700, 3001, 256, 4, 6, 1, 256, 512),
        # a small batch with medium contexts in one layer
        _step("decode_batch8", 1, 8, 16384, 16384, 128, 4, 8, 2, 128, 1024, spans=2),
        # long-document decode: 2 x 59,008 tokens in 16 layers, almost everything Stale
        _step("decode_long_16l", 16, 2, 59008, 59008, 256, 4, 6, 2, 256, 2048),
        # continuous batching: 64 requests of very different lengths
        _step("decode_ragged64", 1, 64, 1024, 131072, 128, 8, 4, 2, 64, 512, spans=3),
        # a large batch before anything has been demoted: FP8 pages only
        _step("decode_fp8_batch32", 1, 32, 32768, 32768, 128, 8, 4, 1, 0, 32768),
        # the long-document step with pages of 1,792 tokens
        _step("decode_blocks_16l", 16, 2, 59008, 59008, 256, 4, 6, 2, 1792, 5 * 1792, spans=3, page=1792),
        # a whole lifecycle step: append, demote one page per request, decode; half of the context Stale
        _step("lifecycle_batch8", 1, 8, 32768, 32768, 128, 8, 4, 2, 0, 16384, retier=True),
        # the retention controller's step: decode with page mass and the score update, in the default format
        _step("scored_batch4", 1, 4, 20011, 40013, 256, 4, 6, 1, 256, 2048, kind="scored"),
        # prefill chunk of several requests, lengths that leave partial pages
        {"name": "append_prefill", "kind": "append", "tokens": 32768 + 77, "requests": 5, "head_dim": 256, "kv_heads": 4,
         "page": 16},
        # a freshly prefilled context ages: thousands of pages to TQ3
        _convert("demote_prefilled", "demote", 3500, 256, 4, 2),
        # an old prefix becomes protected again
        _convert("promote_prefix", "promote", 1023, 128, 8, 1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["scored", "append", "demote", "demote", "promote"])
    d, hkv, group = rng.choice([(128, 1, 8), (128, 4, 8), (128, 8, 4), (128, 8, 4), (256, 4, 6), (256, 4, 6), (256, 2, 4)])
    fmt = rng.choice([1, 2, 2])
    page = rng.choice([16] * 6 + [832, 1792])
    if kind == "append":
        return {"kind": kind, "tokens": _log_int(rng, 40, 131072), "requests": rng.randint(1, 9), "head_dim": d,
                "kv_heads": hkv, "page": page}
    if kind in ("demote", "promote"):
        return {"kind": kind, "pages": max(1, _log_int(rng, 1, 8192) // (page // 16 if page > 16 else 1)), "head_dim": d,
                "kv_heads": hkv, "format": fmt, "page": page}
    layers = rng.choice([1, 1, 4, 16]) if kind == "step" else 1
    batch = _log_int(rng, 1, 64)
    hi = _log_int(rng, 512, 131072)
    lo = hi if rng.random() < 0.5 else max(64, _log_int(rng, max(64, hi // 64), hi))
    while layers * batch * hi * hkv * d > LARGEST:
        if batch > 1:
            batch //= 2
        else:
            hi, lo = hi // 2, max(64, lo // 2)
    anchor = rng.choice([0, 64, 256])
    recent = rng.choice([256, 512, 2048, hi // 2, hi])
    if page > 16:
        anchor, recent = page * rng.choice([0, 1]), page * rng.randint(1, 5)
    return {"kind": kind, "layers": layers, "batch": batch, "ctx_min": min(lo, hi), "ctx_max": hi, "head_dim": d,
            "kv_heads": hkv, "group": group, "format": fmt, "anchor": anchor, "recent": recent,
            "spans": rng.choice([0, 0, 2]), "page": page,
            "retier": kind == "step" and layers == 1 and page == 16 and rng.random() < 0.3}


# ------------------------------------------------------------------------------------------- layout
def _lengths(case):
    """Context lengths of a case: log-spaced from ctx_min to ctx_max, in a fixed shuffled order."""
    n, lo, hi = case["batch"], case["ctx_min"], case["ctx_max"]
    if n == 1:
        return np.array([hi], np.int64)
    x = np.random.RandomState(n).permutation(n) / (n - 1)
    return np.floor(lo * (hi / lo) ** x + 1e-6).astype(np.int64)


def _tags(case, request, length):
    """Tier tag of every page of one request: first tokens Anchor, spans of 128 tokens Anchor, a Recent window at
    the end (all FP8), the rest Stale.  A page that is still open is never Stale."""
    page = case["page"]
    n = -(-length // page)
    tags = np.full(n, M.TAG_STALE, np.uint8)
    first_recent = max(0, length - case["recent"]) // page
    span, rng = max(1, 128 // page), np.random.RandomState(1000 + request)
    for _ in range(case["spans"]):
        if first_recent > span:
            at = rng.randint(0, first_recent - span)
            tags[at:at + span] = M.TAG_ANCHOR
    tags[:case["anchor"] // page] = M.TAG_ANCHOR
    tags[first_recent:] = M.TAG_RECENT
    return tags


def _pages_left(case, lengths):
    """Logical page of every request that leaves the Recent window in this step: its oldest Recent page."""
    return np.maximum(0, lengths - case["recent"]) // case["page"]


def _record_bytes(case):
    d, tiles = case["head_dim"], case["page"] // 16
    return tiles * 32 * d, tiles * (12 * d + 32) + 4 * d           # FP8 page, TQ3 page (one KV head)


# ------------------------------------------------------------------------------------------- inputs
def _generator(seed, stream=0):
    return torch.Generator(device=DEVICE).manual_seed(int(seed) * 101 + stream)


def _kv(gen, tokens, hkv, d, outliers):
    """K and V of some tokens: N(0,1) with a few channels eight times as large, in bf16."""
    k, v = (torch.randn((tokens, hkv, d), generator=gen, device=DEVICE, dtype=torch.bfloat16) for _ in range(2))
    for x, channels in ((k, outliers[0]), (v, outliers[1])):
        x[:, :, channels] *= 8.0
    return k, v


def _outliers(rng, d):
    n = max(1, round(d * 0.02))
    return [torch.from_numpy(np.sort(rng.permutation(d)[:n])).to(DEVICE) for _ in range(2)]


def _filled_pool(case, n_fp8, n_tq3, max_batch, seed, layer):
    """A pool with n_fp8 FP8 and n_tq3 TQ3 pages of random tokens, written by the library's Append and Demote."""
    d, hkv, page = case["head_dim"], case["kv_heads"], case["page"]
    rng, gen = np.random.RandomState((seed * 31 + layer) % (1 << 31)), _generator(seed, layer)
    outliers = _outliers(rng, d)
    stage = max(1, STAGE_TOKENS // page)
    capacity = max(n_fp8, min(n_tq3, stage), 1)
    pool = M.Pool(d, hkv, hkv * case.get("group", 1), capacity, max(n_tq3, 1), rng.randint(0, 2, d) * 2 - 1,
                  max_batch=max_batch, device=DEVICE, page_tokens=page, tq3_format=case.get("format", 1))
    slots = torch.arange(max(stage, 1) * page, dtype=torch.int32, device=DEVICE)
    ids = torch.arange(max(n_tq3, stage), dtype=torch.int32, device=DEVICE)
    for first in range(0, n_tq3, stage):
        n = min(stage, n_tq3 - first)
        pool.append(*_kv(gen, n * page, hkv, d, outliers), slots[:n * page])
        pool.demote(ids[:n], ids[first:first + n].contiguous())
    for first in range(0, capacity, stage):
        n = min(stage, capacity - first)
        pool.append(*_kv(gen, n * page, hkv, d, outliers), slots[:n * page] + first * page)
    return pool, gen, outliers


def _records(pool):
    """The pages of a pool's two arenas, as bytes."""
    n8 = pool.cfg.fp8_pages * pool.hkv * pool.fp8_rec
    n3 = pool.cfg.tq3_pages * pool.hkv * pool.tq3_rec
    return pool.fp8_arena[:n8], pool.tq3_arena[:n3]


def _prepare_decode(case, seed):
    B, d, hkv, group, page = case["batch"], case["head_dim"], case["kv_heads"], case["group"], case["page"]
    hq, rng = hkv * group, np.random.RandomState(seed % (1 << 31))
    lengths = _lengths(case)
    rows = [_tags(case, b, int(n)) for b, n in enumerate(lengths)]
    width = max(len(r) for r in rows)
    tags = np.zeros((B, width), np.uint8)
    used = np.zeros((B, width), bool)
    for b, r in enumerate(rows):
        tags[b, :len(r)] = r
        used[b, :len(r)] = True
    stale = used & (tags == M.TAG_STALE)
    fp8 = used & ~stale
    n_fp8, n_tq3 = int(fp8.sum()), int(stale.sum()) + (B if case["retier"] else 0)
    table = np.full((B, width), -1, np.int32)
    ids3 = rng.permutation(n_tq3).astype(np.int32)
    table[fp8] = rng.permutation(n_fp8).astype(np.int32)
    table[stale] = ids3[:int(stale.sum())]
    last = (lengths - 1) // page
    slots = table[np.arange(B), last] * page + (lengths - 1) % page
    s = {"kind": case["kind"], "scale": d ** -0.5, "page": page,
         "slots": torch.from_numpy(slots.astype(np.int32)).to(DEVICE),
         "lens": torch.from_numpy(lengths.astype(np.int32)).to(DEVICE),
         "pools": [], "bt": [], "tags": [], "q": [], "k": [], "v": [], "out": []}
    for layer in range(case["layers"]):
        pool, gen, outliers = _filled_pool(case, n_fp8, n_tq3, B, seed, layer)
        k, v = _kv(gen, B, hkv, d, outliers)
        s["pools"].append(pool)
        s["bt"].append(torch.from_numpy(table).to(DEVICE))
        s["tags"].append(torch.from_numpy(tags).to(DEVICE))
        s["q"].append(torch.randn((B, hq, d), generator=gen, device=DEVICE, dtype=torch.bfloat16))
        s["k"].append(k)
        s["v"].append(v)
        s["out"].append(torch.zeros((B, hq, d), dtype=torch.float32, device=DEVICE))
    s["result"] = {"out": s["out"], "fp8": [_records(p)[0] for p in s["pools"]]}
    if case["retier"]:
        lp = _pages_left(case, lengths)
        s["src"] = torch.from_numpy(table[np.arange(B), lp]).to(DEVICE)
        s["dst"] = torch.from_numpy(ids3[n_tq3 - B:].copy()).to(DEVICE)
        s["entry"] = torch.from_numpy(np.arange(B) * width + lp).to(DEVICE)
        s["result"].update(tq3=[_records(p)[1] for p in s["pools"]], bt=s["bt"], tags=s["tags"])
    if case["kind"] == "scored":
        s["lse"] = torch.zeros((B, hq), dtype=torch.float32, device=DEVICE)
        s["mass"] = torch.zeros((B, hq, width), dtype=torch.float32, device=DEVICE)
        s["score"] = torch.rand((B, width), generator=gen, device=DEVICE, dtype=torch.float32)
        s["mask"] = (1 << hq) - 1
        s["result"] = {"out": s["out"], "lse": s["lse"], "mass": s["mass"], "score": s["score"]}
    return s


def _prepare_append(case, seed):
    """A prefill chunk of several requests: every request continues somewhere in its own (shuffled) pages."""
    d, hkv, page, n, R = case["head_dim"], case["kv_heads"], case["page"], case["tokens"], case["requests"]
    rng = np.random.RandomState(seed % (1 << 31))
    R = min(R, n)
    cuts = np.linspace(0, n, R + 1).astype(np.int64)
    starts = [0] + [int(np.random.RandomState(r).randint(0, page)) for r in range(1, R)]
    pages = [-(-(starts[r] + int(cuts[r + 1] - cuts[r])) // page) for r in range(R)]
    ids = rng.permutation(sum(pages)).astype(np.int64)
    slots, first = [], 0
    for r in range(R):
        pos = starts[r] + np.arange(cuts[r + 1] - cuts[r])
        slots.append(ids[first + pos // page] * page + pos % page)
        first += pages[r]
    pool = M.Pool(d, hkv, hkv, sum(pages), 1, rng.randint(0, 2, d) * 2 - 1, device=DEVICE, page_tokens=page)
    k, v = _kv(_generator(seed), n, hkv, d, _outliers(rng, d))
    return {"kind": "append", "pool": pool, "k": k, "v": v,
            "slots": torch.from_numpy(np.concatenate(slots).astype(np.int32)).to(DEVICE), "result": _records(pool)[0]}


def _prepare_convert(case, seed):
    """Pages to demote or promote: shuffled sources and destinations, each with its entry in the tables."""
    n, rng = case["pages"], np.random.RandomState(seed % (1 << 31))
    pool, _, _ = _filled_pool(case, n, n, 1, seed, 0)
    ids = [torch.from_numpy(rng.permutation(n).astype(np.int32)).to(DEVICE) for _ in range(2)]
    return {"kind": case["kind"], "pool": pool, "src": ids[0], "dst": ids[1],
            "bt": ids[0].clone(), "tags": torch.full((n,), M.TAG_RECENT if case["kind"] == "demote" else M.TAG_STALE,
                                                     dtype=torch.uint8, device=DEVICE),
            "entry": torch.arange(n, dtype=torch.int64, device=DEVICE), "result": _records(pool)}


def prepare(case, seed):
    if case["kind"] == "append":
        return _prepare_append(case, seed)
    if case["kind"] in ("demote", "promote"):
        return _prepare_convert(case, seed)
    return _prepare_decode(case, seed)


# --------------------------------------------------------------------------------------------- pass
def run(s):
    kind = s["kind"]
    if kind == "append":
        s["pool"].append(s["k"], s["v"], s["slots"])
        return s["result"]
    if kind == "demote":
        s["pool"].demote(s["src"], s["dst"], s["bt"], s["tags"], s["entry"])
        return s["result"][1], s["bt"], s["tags"]
    if kind == "promote":
        s["pool"].promote(s["src"], s["dst"], s["bt"], s["tags"], s["entry"])
        return s["result"][0], s["bt"], s["tags"]
    if kind == "scored":
        s["pools"][0].decode_attention_scored(s["q"][0], s["bt"][0], s["tags"][0], s["lens"], s["scale"], out=s["out"][0],
                                              lse=s["lse"], page_mass=s["mass"])
        M.page_score_update(s["mass"], s["lens"], s["mask"], 0.9, s["score"], page_tokens=s["page"])
        return s["result"]
    if len(s["pools"]) == 1:
        pool = s["pools"][0]
        pool.append(s["k"][0], s["v"][0], s["slots"])
        if "src" in s:
            pool.demote(s["src"], s["dst"], s["bt"][0], s["tags"][0], s["entry"])
        pool.decode_attention(s["q"][0], s["bt"][0], s["tags"][0], s["lens"], s["scale"], out=s["out"][0])
        return s["result"]
    M.append_layers(s["pools"], s["k"], s["v"], s["slots"])
    M.decode_attention_layers(s["pools"], s["q"], s["bt"], s["tags"], s["lens"], s["scale"], s["out"])
    return s["result"]


def work(case):
    d, hkv = case["head_dim"], case["kv_heads"]
    if case["kind"] == "append":
        return {"bytes": case["tokens"] * hkv * 6 * d, "flops": 0}          # bf16 K and V in, e4m3 out
    rec8, rec3 = _record_bytes(case)
    if case["kind"] in ("demote", "promote"):
        return {"bytes": case["pages"] * hkv * (rec8 + rec3), "flops": 0}
    B, hq, lengths = case["batch"], hkv * case["group"], _lengths(case)
    n3 = sum(int((_tags(case, b, int(n)) == M.TAG_STALE).sum()) for b, n in enumerate(lengths))
    pages = sum(-(-int(n) // case["page"]) for n in lengths)
    tokens8 = int(lengths.sum()) - n3 * case["page"]
    nbytes = hkv * (tokens8 * 2 * d + n3 * rec3) + pages * 5 + B * hq * d * 6   # pages, tables, queries, outputs
    if case["kind"] == "scored":
        nbytes += 4 * hq * pages + 8 * pages                                # page mass out, scores in and out
    else:
        nbytes += B * hkv * 6 * d                                           # the appended token
    if case["retier"]:
        nbytes += B * hkv * (rec8 + rec3)
    return {"bytes": case["layers"] * nbytes, "flops": case["layers"] * 4 * d * hq * int(lengths.sum())}


def tolerance(case):
    """Pages and tables are bytes and exact; attention sums are fp32 (scored: with the base-2 logarithm and
    exponential of every page's mass, each good to about 2^-22 of its range)."""
    if case["kind"] in ("append", "demote", "promote"):
        return "exact"
    return {"rel": 2e-5}
