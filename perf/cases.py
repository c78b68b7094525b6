"""Performance cases of the lookup library: what a program that serves from a semantic cache has it do.

A case is one pass through the public entry points (paper_2608_01718_gb300.lacache): a batched lookup (buffers on the
device or on the host, an exact scan or the SimHash index, one lookahead check or an ensemble), a step of the serving
loop, bringing up a cache from a dump of embeddings, or calibrating the thresholds. Inputs are seeded stand-ins for
embeddings: entries in clusters around random unit vectors, queries that are paraphrases of an entry (hits), unrelated
(key misses), or collide with an entry's key under another response prefix (rejections).
"""
from __future__ import annotations

import math

import torch

from paper_2608_01718_gb300 import lacache as L

DEV = "cuda:0"
CHUNK = 1 << 18
CHECKS = {"emb": L.LACACHE_CHECK_EMB, "tokens": L.LACACHE_CHECK_TOKENS, "both": L.LACACHE_CHECK_BOTH}
NEAR_SIGMA, COLL_SIGMA, CLUSTER_SIGMA = 0.05, 0.02, 0.15   # norms of the noise vectors
PERCENTILE, CAP = 5.0, 0.80                                # the key threshold's calibration rule


def _lookup(name, n, d, k, batch, top_c, **kw):
    case = {"name": name, "kind": "lookup", "n": n, "d": d, "k": k, "batch": batch, "top_c": top_c, "tau_c": 0.90,
            "tau_a": 0.80, "check": "emb", "dims": "", "bits": 0, "api": "device", "f32": False, "candidates": False}
    case.update(kw)
    return case


def listed():
    return [
        # the reference cache of a small deployment (an FAQ, one tenant): MiniLM embeddings handed over as fp32, and
        # everything fits in L2, so a batch costs launches and latency
        _lookup("tiny-4k", 4096, 384, 8, 64, 4, tau_c=0.85, f32=True),
        # one user's request at a time, from host memory to host memory, on a mid-sized store of BGE-large embeddings
        _lookup("request-100k", 100_003, 1024, 20, 1, 8, api="host"),
        # a front end's micro-batch against a million entries: the scan is bound by reading the keys
        _lookup("mid-1m", 1 << 20, 768, 16, 32, 8),
        # a full query tile against a large store of BGE-large embeddings
        _lookup("large-4m", 1 << 22, 1024, 16, 128, 8),
        # offline deduplication: thousands of queries at once, a dense contraction on the tensor cores
        _lookup("batch-1m", 1 << 20, 768, 16, 8192, 16, tau_c=0.88),
        # a batch that fills no tile, on an odd store, with both lookahead rules and the candidate lists (what a
        # sharded store's merge or an audit reads)
        _lookup("ragged-300", 300_007, 392, 20, 300, 5, check="both", candidates=True),
        # an ensemble of three lookahead checks (BGE-large, MiniLM and MPNet prefix embeddings)
        _lookup("ensemble-256k", 1 << 18, 768, 16, 32, 8, dims="1024,384,768"),
        # the SimHash index under a small batch (the popcount scan) ...
        _lookup("simhash-1m", 1 << 20, 768, 16, 16, 8, bits=256),
        # ... and under a full one (the tensor-core scan)
        _lookup("simhash-4m", 1 << 22, 768, 16, 128, 8, bits=256),
        # one step of the serving loop: look a batch up, verify the misses' drafts, append the misses
        {"name": "serve-1m", "kind": "serve", "n": 1 << 20, "d": 768, "k": 32, "batch": 256, "top_c": 8,
         "tau_c": 0.90, "tau_a": 0.80},
        # bringing a cache up from a dump of fp32 embeddings: create, insert, index, first lookup
        {"name": "load-512k", "kind": "load", "n": 1 << 19, "d": 768, "k": 16, "batch": 8, "top_c": 8, "tau_c": 0.90,
         "tau_a": 0.80, "bits": 256, "f32": True},
        # threshold calibration on five hundred benign pairs
        {"name": "calibrate-500", "kind": "calibrate", "n": 500, "d": 1024},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: at most 8 GB of keys, at most the work of batch-1m."""
    kind = rng.choice(["lookup"] * 5 + ["simhash"] * 3 + ["serve", "load", "calibrate"])
    d = 8 * _log(rng, 16, 160)
    k = _log(rng, 4, 64)
    top_c = _log(rng, 1, 32)
    check = rng.choice(["emb", "emb", "tokens", "both"])
    if kind == "lookup":
        n = _log(rng, 1000, min(1 << 22, (1 << 32) // d))
        batch = min(_log(rng, 1, 8192), max(1, (1 << 42) // (n * d)))
        dims = rng.choice(["", "", "", "384,768", "1024,384,768"])
        api = "device" if dims else rng.choice(["device", "device", "device", "host", "noalloc"])
        return {**_lookup("", n, d, k, batch, top_c, check=check, dims=dims, api=api,
                          f32=n < 100_000 and rng.random() < 0.3, candidates=rng.random() < 0.3), "name": "drawn"}
    if kind == "simhash":
        bits = rng.choice([128, 256, 512])
        n = _log(rng, 20_000, min(1 << 22, (1 << 32) // d))
        return {**_lookup("", n, d, k, _log(rng, 1, 400), top_c, check=check, bits=bits,
                          api=rng.choice(["device", "device", "host"])), "name": "drawn"}
    if kind == "serve":
        return {"name": "drawn", "kind": "serve", "n": _log(rng, 100_000, 1 << 20), "d": d, "k": k,
                "batch": _log(rng, 16, 512), "top_c": top_c, "tau_c": 0.90, "tau_a": 0.80}
    if kind == "load":
        return {"name": "drawn", "kind": "load", "n": _log(rng, 20_000, (1 << 29) // d), "d": d, "k": k,
                "batch": _log(rng, 1, 64), "top_c": top_c, "tau_c": 0.90, "tau_a": 0.80,
                "bits": rng.choice([0, 128, 256, 512]), "f32": rng.random() < 0.6}
    return {"name": "drawn", "kind": "calibrate", "n": _log(rng, 100, min(1 << 21, (1 << 30) // d)), "d": d}


# ---- inputs -------------------------------------------------------------------------------------------------------

def _gen(seed, tag):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1009 + tag)
    return g


def _randn(rows, d, g):
    return torch.randn((rows, d), generator=g, device=DEV)


def _unit(x):
    return x / x.norm(dim=1, keepdim=True)


def _unit_rows(rows, dims, g):
    """One unit vector per model, back to back."""
    return torch.cat([_unit(_randn(rows, dim, g)) for dim in dims], dim=1)


def _dims(case):
    text = case.get("dims", "")
    return [int(x) for x in text.split(",")] if text else [case["d"]]


def _store(case, seed):
    """The entries: key rows, prefix rows (bf16, or fp32 for a case that hands those over) and token ids."""
    n, d, dims = case["n"], case["d"], _dims(case)
    dtype = torch.float32 if case.get("f32") else torch.bfloat16
    g = _gen(seed, 1)
    clusters = min(4096, max(1, n // 64))
    centres = _unit(_randn(clusters, d, g))
    key = torch.empty((n, d), dtype=dtype, device=DEV)
    prefix = torch.empty((n, sum(dims)), dtype=dtype, device=DEV)
    for j in range(0, n, CHUNK):
        rows = min(CHUNK, n - j)
        at = torch.randint(0, clusters, (rows,), generator=g, device=DEV)
        key[j:j + rows] = _unit(centres[at] + _randn(rows, d, g) * (CLUSTER_SIGMA / math.sqrt(d)))
        prefix[j:j + rows] = _unit_rows(rows, dims, g)
    ids = torch.randint(0, 128256, (n, case["k"]), generator=g, device=DEV, dtype=torch.int32)
    return key, prefix, ids


def _queries(case, seed, store, batches=1):
    """`batches` batches of queries: about half paraphrases of an entry, three tenths unrelated, the rest collisions."""
    key, prefix, ids = store
    rows, d = case["batch"] * batches, case["d"]
    g = _gen(seed, 2)
    u = torch.rand((rows, 1), generator=g, device=DEV)
    near, unrelated = u < 0.5, u >= 0.7
    target = torch.randint(0, case["n"], (rows,), generator=g, device=DEV)
    sigma = torch.where(near, NEAR_SIGMA, COLL_SIGMA) / math.sqrt(d)
    emb = _unit(torch.where(unrelated, _randn(rows, d, g), key[target].float() + _randn(rows, d, g) * sigma))
    fresh = _unit_rows(rows, _dims(case), g).bfloat16()
    fresh_ids = torch.randint(0, 128256, (rows, case["k"]), generator=g, device=DEV, dtype=torch.int32)
    return (emb.bfloat16().contiguous(), torch.where(near, prefix[target].bfloat16(), fresh).contiguous(),
            torch.where(near, ids[target], fresh_ids).contiguous())


def _serve_batches(case):
    # enough batches that a long run of passes still brings new queries
    return max(4, 512_000 // case["batch"])


def _serve_queries(case, seed, store):
    """The serving loop's batches. The last tenth of a batch repeats the first queries of the batch before it, whose
    misses are entries by then."""
    b, t = case["batch"], max(1, case["batch"] // 10)
    out = []
    for x in _queries(case, seed, store, _serve_batches(case)):
        x = x.view(-1, b, x.shape[1])
        x[1:, b - t:] = x[:-1, :t].clone()
        out.append(x)
    return out


def _radius(tau_c, bits):
    """Keeps an entry at the key threshold with a probability of about Phi(4)."""
    p = math.acos(tau_c) / math.pi
    return min(bits, math.ceil(bits * p + 4.0 * math.sqrt(bits * p * (1 - p))))


def _hyperplanes(case, seed):
    return _randn(case["bits"], case["d"], _gen(seed, 3)).bfloat16()


def _pairs(case, seed):
    g = _gen(seed, 4)
    x = torch.empty((case["n"], case["d"]), dtype=torch.bfloat16, device=DEV)
    y = torch.empty_like(x)
    for j in range(0, case["n"], CHUNK):
        rows = min(CHUNK, case["n"] - j)
        a = _unit(_randn(rows, case["d"], g))
        x[j:j + rows] = a
        y[j:j + rows] = _unit(a + _randn(rows, case["d"], g) * (0.6 / math.sqrt(case["d"])))
    return x, y


# ---- a pass -------------------------------------------------------------------------------------------------------

def _cache(case, capacity):
    dims = _dims(case)
    many = {"prefix_dims": dims, "tau_a_models": [0.7] * len(dims)} if case.get("dims") else {}
    return L.LaCache(case["d"], case["k"], capacity, case["tau_c"], case["tau_a"], case["top_c"],
                     max_batch=case["batch"], check_mode=CHECKS[case.get("check", "emb")],
                     token_match_min=(case["k"] + 1) // 2,
                     stage1=L.LACACHE_STAGE1_LSH if case.get("bits") else L.LACACHE_STAGE1_AUTO, **many)


def _insert(cache, case, store):
    cache.insert(*store, dtype=L.LACACHE_F32 if case.get("f32") else L.LACACHE_BF16)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "calibrate":
        x, y = _pairs(case, seed)
        return {"kind": kind, "x": x, "y": y, "sims": torch.empty(case["n"], device=DEV),
                "result": torch.empty(2, device=DEV),
                "workspace": torch.empty(L.lacache_calibrate_workspace_bytes(), dtype=torch.uint8, device=DEV)}
    store = _store(case, seed)
    if kind == "load":
        return {"kind": kind, "case": case, "store": store, "queries": _queries(case, seed, store),
                "hyper": _hyperplanes(case, seed) if case["bits"] else None,
                "radius": _radius(case["tau_c"], case["bits"]) if case["bits"] else 0,
                "sig": torch.empty((case["n"], case["bits"] // 32), dtype=torch.int32, device=DEV),
                "out": L.alloc_result(case["batch"], case["top_c"], DEV, candidates=False)}
    if kind == "serve":
        batches = _serve_batches(case)
        cache = _cache(case, case["n"] + batches * case["batch"])
        _insert(cache, case, store)
        g = _gen(seed, 5)
        draft = torch.rand((case["batch"], case["k"]), generator=g, device=DEV)
        target = (draft + 0.2 * torch.randn(draft.shape, generator=g, device=DEV) + 0.3).clamp(0.0, 1.0)
        return {"kind": kind, "cache": cache, "queries": _serve_queries(case, seed, store), "at": 0, "batches": batches,
                "target": target, "draft": draft,
                "accepted": torch.empty(case["batch"], dtype=torch.int32, device=DEV),
                "out": L.alloc_result(case["batch"], case["top_c"], DEV, candidates=False)}
    queries = _queries(case, seed, store)
    models = len(_dims(case))
    if case["api"] == "noalloc":
        store = tuple(x if i == 2 else x.bfloat16() for i, x in enumerate(store))
        cfg = L.make_config(case["d"], case["k"], case["n"], case["tau_c"], case["tau_a"], case["top_c"],
                            max_batch=case["batch"], check_mode=CHECKS[case["check"]],
                            token_match_min=(case["k"] + 1) // 2)
        return {"kind": "noalloc", "cfg": cfg, "store": store, "queries": queries,
                "out": L.alloc_result(case["batch"], case["top_c"], DEV, candidates=case["candidates"])}
    cache = _cache(case, case["n"])
    _insert(cache, case, store)
    if case["bits"]:
        L.lacache_enable_lsh(cache.h, case["bits"], _radius(case["tau_c"], case["bits"]), _hyperplanes(case, seed))
    host = case["api"] == "host"
    if host:
        queries = tuple(x.cpu().pin_memory() for x in queries)
    return {"kind": case["api"], "cache": cache, "queries": queries,
            "out": L.alloc_result(case["batch"], case["top_c"], "cpu" if host else DEV, candidates=case["candidates"],
                                  pinned=host, models=models if case["dims"] else 0)}


def run(s):
    kind = s["kind"]
    if kind == "device":
        return s["cache"].lookup(*s["queries"], out=s["out"])
    if kind == "host":
        L.lacache_lookup_host(s["cache"].h, *s["queries"], s["out"])
        return s["out"]
    if kind == "noalloc":
        L.lacache_lookup_noalloc(s["cfg"], *s["store"], *s["queries"], s["out"])
        return s["out"]
    if kind == "serve":
        emb, prefix, ids = (x[s["at"]] for x in s["queries"])
        s["at"] = (s["at"] + 1) % s["batches"]
        cache, out = s["cache"], s["out"]
        cache.lookup(emb, prefix, ids, out=out)
        L.lacache_verify_draft(s["target"], s["draft"], out["status"], s["accepted"])
        first, appended = cache.append_misses(emb, prefix, ids, out["status"])
        return {**out, "accepted": s["accepted"], "first": first, "appended": appended}
    if kind == "load":
        case = s["case"]
        with _cache(case, case["n"]) as cache:
            _insert(cache, case, s["store"])
            if case["bits"]:
                L.lacache_enable_lsh(cache.h, case["bits"], s["radius"], s["hyper"])
                L.lacache_read_signatures(cache.h, 0, case["n"], s["sig"])
            cache.lookup(*s["queries"], out=s["out"])
        return {**s["out"], "sig": s["sig"]}
    L.lacache_calibrate(s["x"], s["y"], PERCENTILE, CAP, s["sims"], s["result"], s["workspace"])
    return {"sims": s["sims"], "result": s["result"]}


def work(case):
    n, d = case["n"], case["d"]
    if case["kind"] == "calibrate":
        return {"bytes": 4 * n * d + 4 * n, "flops": 2 * n * d}
    b, k, c, pd, bits = case["batch"], case["k"], case["top_c"], sum(_dims(case)), case.get("bits", 0)
    row = 2 * d + 2 * pd + 4 * k
    queries, gathered = b * row, 0.7 * b * c * (2 * pd + 4 * k)   # three queries in ten have no candidate
    related = 0.7 * b * n / min(4096, max(1, n // 64))            # (query, entry) pairs of one cluster
    if case["kind"] == "load":
        given = n * (4 * (d + pd) + 4 * k if case["f32"] else row)
        return {"bytes": given + n * row + queries + gathered + (n * bits / 8 + 2 * bits * d if bits else 2 * n * d),
                "flops": 2 * n * d * (bits or b)}
    if bits:
        return {"bytes": n * bits / 8 + 2 * bits * d + queries + gathered + min(related, n) * 2 * d,
                "flops": 2 * b * d * bits + 2 * related * d}
    appended = 0.5 * b * 2 * row if case["kind"] == "serve" else 0
    return {"bytes": 2 * n * d + queries + gathered + appended, "flops": 2 * b * n * d}


def tolerance(case):
    # scores are fp32 sums of exact bf16 products; candidates within rounding of one another may change places, and
    # with them the entry, prefix score and token count shown in a slot of the candidate list
    if case.get("candidates"):
        return {"rel": 0.03, "max": 0.99, "differ": 0.01}
    return {"rel": 1e-5, "max": 1e-4, "differ": 1e-3}


# ---- the same in 64 bits --------------------------------------------------------------------------------------------

def _dots(a, b, dims):
    """Every model's dot product of two rows of prefix embeddings, [rows x models]."""
    return torch.stack([(x * y).sum(-1) for x, y in zip(a.split(dims, -1), b.split(dims, -1))], -1)


def _decide(case, store, queries):
    """The lookup of Algorithm 1 in 64 bits: per query the first top_c entries with a key score of at least tau_c, and
    of them the first whose prefix passes."""
    key, prefix, ids = (x if x.dtype == torch.int32 else x.bfloat16() for x in store)
    emb, qprefix, qids = queries
    n, c, dims = case["n"], case["top_c"], _dims(case)
    m = len(dims)
    tau_c = float(torch.tensor(case["tau_c"]))
    taus = torch.tensor([0.7] * m if case.get("dims") else [case["tau_a"]], device=DEV).double()
    parts = []
    for q0 in range(0, emb.shape[0], 512):
        e = emb[q0:q0 + 512].double()
        top = torch.full((e.shape[0], 0), 0.0, device=DEV, dtype=torch.float64)
        at = torch.zeros((e.shape[0], 0), device=DEV, dtype=torch.int64)
        for j in range(0, n, CHUNK):
            s = e @ key[j:j + CHUNK].double().T
            v, i = s.topk(min(c, s.shape[1]), dim=1)
            top, at = torch.cat([top, v], 1), torch.cat([at, i + j], 1)
            top, o = top.sort(dim=1, descending=True, stable=True)
            top, at = top[:, :c], at.gather(1, o)[:, :c]
        if top.shape[1] < c:   # a store of fewer than c entries
            fill = c - top.shape[1]
            top = torch.nn.functional.pad(top, (0, fill), value=-2.0)
            at = torch.nn.functional.pad(at, (0, fill))
        valid = top >= tau_c
        r = _dots(qprefix[q0:q0 + 512, None].double(), prefix[at].double(), dims)
        match = (qids[q0:q0 + 512, None] == ids[at]).sum(-1)
        emb_ok, tok_ok = (r >= taus).all(-1), match >= (case["k"] + 1) // 2
        ok = {"emb": emb_ok, "tokens": tok_ok, "both": emb_ok & tok_ok}[case.get("check", "emb")] & valid
        hit, first = ok.any(1), ok.int().argmax(1)
        shown = torch.where(hit, first, 0)[:, None]
        nan = torch.full_like(top, float("nan"))
        one = torch.where(valid[:, 0], r[..., 0].gather(1, shown)[:, 0], nan[:, 0])
        score = torch.where(hit, top.gather(1, shown)[:, 0], top[:, 0])
        shown_r = r.gather(1, shown[..., None].expand(-1, -1, m))[:, 0]
        parts.append({"key_score": score, "prefix_score": one, "cand_score": torch.where(valid, top, nan),
                      "cand_prefix_score": torch.where(valid, r[..., 0], nan),
                      "prefix_scores": torch.where(valid[:, :1], shown_r, nan[:, :1])})
    return {name: torch.cat([p[name] for p in parts]) for name in parts[0]}


def exact(case, seed):
    if case["kind"] == "calibrate":
        x, y = _pairs(case, seed)
        sims = torch.cat([(x[j:j + CHUNK].double() * y[j:j + CHUNK].double()).sum(1)
                          for j in range(0, case["n"], CHUNK)])
        rank = min(case["n"], max(1, math.ceil(PERCENTILE / 100.0 * case["n"])))
        value = sims.sort().values[rank - 1]
        return {"sims": sims, "result": torch.stack([value, value.clamp(max=CAP)])}
    if 2.0 * case["batch"] * case["n"] * case["d"] > 1.4e13:
        return None   # over ten seconds in 64 bits
    store = _store(case, seed)
    queries = [x[0] for x in _serve_queries(case, seed, store)] if case["kind"] == "serve" \
        else _queries(case, seed, store)
    want = _decide(case, store, queries)
    names = ["entry_id", "status", "key_score", "prefix_score", "token_matches", "n_cand"]
    if case.get("candidates"):
        names += ["cand_id", "cand_score", "cand_prefix_score", "cand_matches", "cand_pass"]
    if case.get("dims"):
        names += ["prefix_scores"]
    if case.get("bits"):
        want.pop("key_score")   # a miss reports the best admitted entry, which the index decides
    return {name: want.get(name) for name in names}
