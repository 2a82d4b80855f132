"""The work that users of this library have it do, as measurable cases.

A case is a dict of plain values; `prepare` makes, from a seed, what a program
holds before the call (an index, a cross model, the request's arrays, the
result buffers), `run` is one pass through the public entry points, `work` the
bytes and operations that pass cannot do without, and `exact` the same results
in 64 bits from plain torch operations.

Sizes follow this repository's own recipes (datagen.RECIPES, bench.py).  The
inputs are drawn on the GPU with torch, from the same distributions: N(0, 1/d)
embeddings, heavy-tailed (finite Zipf) categorical fields over vocabularies
spread over [10, 100000] on a logarithmic scale or of one fixed size, normal
cross weights, targeting bitmaps of a random density.
"""
import math

import numpy as np
import torch

from paper_2511_22460_gb300 import ebr

DEV = torch.device("cuda", 0)
HASH_BITS = 24

# Values every case starts from.  op: what is called ("topk": score_topk;
# "noalloc": scan_topk_noalloc; "build": build_index and the first scores of
# the new index).  vocab 0: log-spaced sizes in [10, 100000], else that size.
# n_keys_q: keys of a sparse key list (0: the request carries user fields).
# history: most values of a multi-valued user field (0: one value each).
# empty: share of (ad, field) entries without a value.
_BASE = {"op": "topk", "n_ads": 0, "d": 64, "dtype": "f32", "fields": 16, "vocab": 0,
         "zipf": 1.05, "pairs": 64, "dense_w": False, "w_var": 0.05, "k": 500, "batch": 1,
         "mixed_k": False, "filter": False, "history": 0, "empty": 0.0, "n_keys_q": 0,
         "host": False}


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # a small inventory: launches and latency are all of it
        _case("topk_fp32_10k", n_ads=10_000, d=32, fields=4, vocab=50, zipf=1.1, pairs=16,
              dense_w=True, w_var=0.1, k=100),
        # an ordinary inventory of one advertiser category
        _case("topk_fp32_200k", n_ads=200_000, k=500),
        # the plain FP32 request at inventory scale (the default benchmark)
        _case("topk_fp32_2m", n_ads=2_000_000, k=500),
        # the paper's regime: a user's history touches a few popular keys
        _case("sparse30_fp32_2m", n_ads=2_000_000, k=100, n_keys_q=30),
        _case("sparse300_fp32_2m", n_ads=2_000_000, k=500, n_keys_q=300),
        # one request from host buffers: user histories, a targeting bitmap,
        # ads that lack some features, odd sizes
        _case("topk_bf16_host_1m", n_ads=1_000_003, d=128, dtype="bf16", fields=24, pairs=96,
              k=137, filter=True, history=8, empty=0.1, host=True),
        # the largest single request: 10M FP8 rows, 32 keys per ad
        _case("topk_fp8_10m", n_ads=10_000_000, dtype="fp8e4m3", fields=32, vocab=15, zipf=1.0,
              pairs=128, k=2000),
        # offline / peak-load batches
        _case("batch256_bf16_5m", n_ads=5_000_000, d=128, dtype="bf16", fields=24, pairs=96,
              k=1000, batch=256),
        _case("batch64_fp8_10m", n_ads=10_000_000, dtype="fp8e4m3", fields=32, vocab=15,
              zipf=1.0, pairs=128, k=2000, batch=64),
        # a full serving wave: K and targeting bitmap per request
        _case("wave128_bf16_5m", n_ads=5_000_000, dtype="bf16", fields=32, pairs=128, k=2000,
              batch=128, mixed_k=True, filter=True),
        # the periodic rebuild of the index, up to the first scores it gives
        _case("build_fp32_2m", op="build", n_ads=2_000_000),
        # the allocation-free scan over the caller's own buffers, a ragged size
        _case("noalloc_fp32_777k", op="noalloc", n_ads=777_777, d=128, fields=1, pairs=1, k=500,
              filter=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["topk", "topk", "topk", "sparse", "batch", "batch", "build", "noalloc"])
    fields = rng.randint(4, 32)
    c = {"fields": fields, "pairs": rng.randint(fields, min(4 * fields, fields * fields)),
         "vocab": rng.choice([0, 0, 15, 300]), "zipf": round(rng.uniform(1.0, 1.2), 3)}
    if kind == "noalloc":
        return _case(op="noalloc", n_ads=_log_int(rng, 5_000, 3_000_000),
                     d=rng.choice([4, 8, 16, 32, 64, 128]), fields=1, pairs=1,
                     k=_log_int(rng, 1, 1024), filter=rng.random() < 0.5)
    if kind == "build":
        return _case(op="build", n_ads=_log_int(rng, 20_000, 2_000_000),
                     d=rng.choice([16, 32, 64]), dtype=rng.choice(["f32", "bf16", "fp8e4m3"]),
                     empty=rng.choice([0.0, 0.1]), **c)
    if kind == "sparse":
        return _case(n_ads=_log_int(rng, 50_000, 3_000_000), d=rng.choice([16, 32, 64, 128]),
                     dtype=rng.choice(["f32", "bf16"]), k=_log_int(rng, 10, 100),
                     n_keys_q=_log_int(rng, 3, 3000), host=rng.random() < 0.25, **c)
    if kind == "batch":
        batch = _log_int(rng, 60, 256)
        c["fields"] = rng.randint(16, 32)
        c["pairs"] = rng.randint(c["fields"], 4 * c["fields"])
        return _case(n_ads=_log_int(rng, 50_000, 100_000_000 // batch),
                     d=rng.choice([64, 128]), dtype=rng.choice(["bf16", "fp8e4m3"]),
                     k=rng.choice([1500, 2000]), batch=batch, filter=rng.random() < 0.5,
                     history=rng.choice([0, 0, 6]), empty=rng.choice([0.0, 0.1]),
                     host=rng.random() < 0.25, **c)
    return _case(n_ads=_log_int(rng, 5_000, 4_000_000), d=rng.choice([16, 32, 64, 128]),
                 dtype=rng.choice(["f32", "f32", "bf16", "fp8e4m3"]), k=_log_int(rng, 10, 2000),
                 filter=rng.random() < 0.4, history=rng.choice([0, 0, 6]),
                 empty=rng.choice([0.0, 0.1]), host=rng.random() < 0.25, **c)


# ------------------------------------------------------------------- inputs
def _vocabs(c):
    f = c["fields"]
    if c["vocab"]:
        return np.full(f, c["vocab"], np.int64)
    q = (np.arange(f) + 0.5) / f
    return np.rint(np.exp(math.log(10) + q * (math.log(100_000) - math.log(10)))).astype(np.int64)


def _zipf(g, V, s, n):
    """n values of 0..V-1, P(rank r) ~ r^-s, ranks mapped to values at random."""
    cdf = torch.cumsum(torch.arange(1, V + 1, device=DEV, dtype=torch.float64) ** -s, 0)
    cdf /= cdf[-1].clone()
    r = torch.searchsorted(cdf, torch.rand(n, device=DEV, dtype=torch.float64, generator=g))
    perm = torch.randperm(V, device=DEV, generator=g, dtype=torch.int64)
    return perm[r.clamp_(max=V - 1)].to(torch.int32)


def _bitmaps(g, n, fracs):
    """[len(fracs), ceil(n / 64)] int64 words, bit a of word a >> 6 set with that probability."""
    words = (n + 63) // 64
    out = torch.empty((len(fracs), words), dtype=torch.int64, device=DEV)
    sh = torch.arange(64, device=DEV, dtype=torch.int64)
    for b, f in enumerate(fracs):
        bits = torch.rand(words * 64, device=DEV, generator=g) < f
        bits[n:] = False
        out[b] = (bits.view(words, 64).to(torch.int64) << sh).sum(1)
    return out


def _inputs(c, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    rng = np.random.default_rng(seed)
    n, d, f, B = c["n_ads"], c["d"], c["fields"], c["batch"]
    x = {}
    x["emb"] = torch.randn((n, d), device=DEV, generator=g) * (1.0 / math.sqrt(d))
    x["h_u"] = torch.randn((B, d), device=DEV, generator=g) * (1.0 / math.sqrt(d))
    x["ks"] = [c["k"]] * B
    if c["mixed_k"]:
        x["ks"] = [int(v) for v in rng.choice([max(1, c["k"] // 10), max(1, c["k"] // 2), c["k"]], B)]
        x["ks"][0] = c["k"]
    x["ks"] = [min(k, n) for k in x["ks"]]
    x["filter"] = _bitmaps(g, n, rng.uniform(0.01 if B > 1 else 0.2, 1.0, B)) if c["filter"] else None
    if c["op"] == "noalloc":
        x["wide"] = torch.randn(n, device=DEV, generator=g)
        return x
    V = _vocabs(c)
    off = np.concatenate([[0], np.cumsum(V)])
    x["vocab"], x["n_keys"] = V, int(off[-1])
    # the ads' keys (-1: no value in that field)
    ad_key = torch.empty((n, f), dtype=torch.int32, device=DEV)
    for j in range(f):
        ad_key[:, j] = _zipf(g, int(V[j]), c["zipf"], n) + int(off[j])
    if c["empty"]:
        for j in range(f):
            ad_key[torch.rand(n, device=DEV, generator=g) < c["empty"], j] = -1
    x["ad_key"] = ad_key
    pairs = np.array([(i, j) for i in range(f) for j in range(f)], np.uint32)
    if c["pairs"] < len(pairs):
        pairs = pairs[np.sort(rng.choice(len(pairs), c["pairs"], replace=False))]
    x["pairs"] = pairs
    if c["dense_w"]:
        sizes = [int(V[i] * V[j]) for i, j in pairs]
        x["w_off"] = np.concatenate([[0], np.cumsum(sizes)])[:-1].astype(np.uint64)
        x["w"] = torch.randn(sum(sizes), device=DEV, generator=g) * math.sqrt(c["w_var"])
    else:
        x["w_off"] = None
        x["w"] = torch.randn(1 << HASH_BITS, device=DEV, generator=g) * math.sqrt(c["w_var"])
    # the users: one value per field, or a history of 0..history of them
    x["users"] = []
    cols = [_zipf(g, int(V[i]), c["zipf"], B * max(1, c["history"])).cpu().numpy() for i in range(f)]
    for b in range(B):
        if not c["history"]:
            x["users"].append((None, np.array([cols[i][b] for i in range(f)], np.uint32)))
            continue
        lens = rng.integers(1, c["history"] + 1, f)
        lens[rng.random(f) < 0.1] = 0
        ptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint32)
        vals = np.concatenate([cols[i][b * c["history"]:b * c["history"] + lens[i]]
                               for i in range(f)]).astype(np.uint32)
        x["users"].append((ptr, vals))
    x["q_key"] = None
    if c["n_keys_q"]:
        # keys drawn in proportion to their posting lists
        pick = torch.randint(0, n * f, (4 * c["n_keys_q"],), device=DEV, generator=g)
        key = ad_key.view(-1)[pick].cpu().numpy()
        _, first = np.unique(key, return_index=True)
        x["q_key"] = key[np.sort(first)][:c["n_keys_q"]].astype(np.uint32)
        x["q_w"] = (rng.standard_normal(x["q_key"].size) * math.sqrt(c["w_var"])).astype(np.float32)
    return x


def _postings(c, x):
    n, f = x["ad_key"].shape
    key = x["ad_key"].reshape(-1)
    ad = torch.arange(n, device=DEV, dtype=torch.int32).repeat_interleave(f)
    if c["empty"]:
        has = key >= 0
        key, ad = key[has], ad[has]
    return key.contiguous(), ad.contiguous()


def _cross(x):
    return ebr.cross_create(x["vocab"], x["vocab"], x["pairs"], x["w"], x["w_off"],
                            hashed=x["w_off"] is None, hash_bits=HASH_BITS)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).to(DEV)


def prepare(case, seed):
    c, x = case, _inputs(case, seed)
    B, kmax = c["batch"], max(x["ks"])
    s = {"case": c}
    if c["op"] == "noalloc":
        s.update(emb=x["emb"], h_u=x["h_u"][0].clone(), wide=x["wide"], k=x["ks"][0],
                 filter=None if x["filter"] is None else x["filter"][0].clone(),
                 ids=torch.empty(kmax, dtype=torch.int32, device=DEV),
                 scores=torch.empty(kmax, device=DEV))
        return s
    s["cross"] = _cross(x)
    key, ad = _postings(c, x)
    del x["ad_key"]
    if c["op"] == "build":
        s.update(key=key, ad=ad, emb=x["emb"], n_keys=x["n_keys"],
                 query=ebr.Query(h_u=x["h_u"][0].clone(), k=x["ks"][0],
                                 user_vals=_dev(x["users"][0][1])))
        return s
    s["index"] = ebr.build_index(c["n_ads"], x["n_keys"], key, ad, x["emb"], dtype=c["dtype"])
    del key, ad, x["emb"]
    host = c["host"]
    put = (lambda a: np.ascontiguousarray(a)) if host else _dev
    h_u = x["h_u"].cpu().numpy() if host else x["h_u"]
    filt = x["filter"]
    if filt is not None and host:
        filt = filt.cpu().numpy().view(np.uint64)
    s["queries"] = []
    for b in range(B):
        q = {"h_u": h_u[b].copy() if host else h_u[b].clone(), "k": x["ks"][b],
             "filter": None if filt is None else (filt[b].copy() if host else filt[b].clone())}
        if x["q_key"] is not None:
            q.update(q_key=put(x["q_key"]),
                     q_w=x["q_w"] if host else torch.from_numpy(x["q_w"]).to(DEV))
        else:
            ptr, vals = x["users"][b]
            q.update(user_vals=put(vals), user_ptr=None if ptr is None else put(ptr))
        s["queries"].append(ebr.Query(**q))
    if host:
        s.update(ids=np.empty((B, kmax), np.uint32), scores=np.empty((B, kmax), np.float32))
    else:
        s.update(ids=torch.empty((B, kmax), dtype=torch.int32, device=DEV),
                 scores=torch.empty((B, kmax), device=DEV))
    return s


# --------------------------------------------------------------------- pass
def run(state):
    s, c = state, state["case"]
    if c["op"] == "noalloc":
        ebr.scan_topk_noalloc(s["emb"], s["h_u"], s["wide"], s["filter"], s["k"], s["ids"],
                              s["scores"])
        return {"ids": s["ids"], "scores": s["scores"]}
    if c["op"] == "build":
        ix = ebr.build_index(c["n_ads"], s["n_keys"], s["key"], s["ad"], s["emb"],
                             dtype=c["dtype"])
        scores = torch.empty(c["n_ads"], device=DEV)
        wide = torch.empty(c["n_ads"], device=DEV)
        ebr.score_all(ix, s["cross"], s["query"], scores)
        ebr.wide_scores(ix, s["cross"], s["query"], wide)
        i = ix.info()
        info = [i.nnz_unique, i.index_bytes, i.emb_bytes, i.window_view_bytes, i.n_windows,
                i.max_keys_per_ad, i.max_window_slots] + list(i.n_blocks)
        ix.close()
        return {"scores": scores, "wide": wide, "info": np.array(info, np.int64)}
    ebr.score_topk(s["index"], s["cross"], s["queries"], s["ids"], s["scores"],
                   io=ebr.IO_HOST if c["host"] else ebr.IO_DEVICE)
    return {"ids": s["ids"], "scores": s["scores"]}


def work(case):
    """The table and the postings (one byte each, the inverted list's own
    value bytes) are read once, the results written once."""
    c = case
    n, d, f, B = c["n_ads"], c["d"], c["fields"], c["batch"]
    row = d * {"f32": 4, "bf16": 2, "fp8e4m3": 1}[c["dtype"]] + (4 if c["dtype"] == "fp8e4m3" else 0)
    if c["op"] == "noalloc":
        return {"bytes": n * (row + 4) + (n // 8 if c["filter"] else 0) + 8 * c["k"],
                "flops": 2 * n * d + n}
    nnz = n * f * (1.0 - c["empty"])
    if c["op"] == "build":
        # pairs and vectors in, the list (value bytes) and the table out, two score vectors
        return {"bytes": 8 * nnz + 4 * n * d + nnz + n * row + 8 * n, "flops": 2 * n * d + 2 * nnz}
    adds = nnz
    if c["n_keys_q"]:
        # expected postings of the listed keys: their share of the key space at least
        V = _vocabs(c)
        adds = nnz * min(1.0, c["n_keys_q"] / float(V.sum()))
    return {"bytes": n * row + adds + B * (8 * c["k"] + (n // 8 if c["filter"] else 0)),
            "flops": B * (2.0 * n * d + adds)}


# -------------------------------------------------------------- in 64 bits
def _splitmix_index(p, u, v):
    """splitmix64((p << 40) | (u << 20) | v) & (2^24 - 1); v: int64 tensor."""
    def lsr(z, s):
        return (z >> s) & ((1 << (64 - s)) - 1)

    def const(k):
        return k - (1 << 64) if k >= 1 << 63 else k
    z = (v | ((int(p) << 40) | (int(u) << 20))) + const(0x9E3779B97F4A7C15)
    z = (z ^ lsr(z, 30)) * const(0xBF58476D1CE4E5B9)
    z = (z ^ lsr(z, 27)) * const(0x94D049BB133111EB)
    return (z ^ lsr(z, 31)) & ((1 << HASH_BITS) - 1)


def _expand64(x, b):
    """The expanded weights of user b over the key space, float64, and a last 0."""
    V = x["vocab"]
    off = np.concatenate([[0], np.cumsum(V)])
    w = torch.zeros(x["n_keys"] + 1, dtype=torch.float64, device=DEV)
    if x["q_key"] is not None:
        key = torch.from_numpy(x["q_key"].astype(np.int64)).to(DEV)
        w.index_add_(0, key, torch.from_numpy(x["q_w"]).to(DEV).double())
        return w
    ptr, vals = x["users"][b]
    for p, (i, j) in enumerate(x["pairs"].tolist()):
        us = vals[i:i + 1] if ptr is None else vals[ptr[i]:ptr[i + 1]]
        v = torch.arange(int(V[j]), device=DEV, dtype=torch.int64)
        for u in us.tolist():
            if x["w_off"] is None:
                t = x["w"][_splitmix_index(p, u, v)]
            else:
                o = int(x["w_off"][p]) + u * int(V[j])
                t = x["w"][o:o + int(V[j])]
            w[int(off[j]):int(off[j + 1])] += t.double()
    return w


def _masked(score, words, a0):
    """score [m] of ads a0.. (a0 a multiple of 64) with -inf where the bitmap is 0."""
    m = score.numel()
    wd = words[a0 // 64:(a0 + m + 63) // 64]
    bit = (wd[:, None] >> torch.arange(64, device=DEV, dtype=torch.int64)) & 1
    return torch.where(bit.view(-1)[:m] == 1, score, -math.inf)


def exact(case, seed):
    c, x = case, _inputs(case, seed)
    n, f, B, ks = c["n_ads"], c["fields"], c["batch"], x["ks"]
    kmax = max(ks)
    h = x["h_u"].double()
    wts = None
    if c["op"] != "noalloc":
        wts = torch.stack([_expand64(x, b) for b in range(B)], 1)  # [n_keys + 1][B]
    step = max(64, (1 << 26) // max(B, c["d"]) // 64 * 64)
    best_s = torch.full((B, kmax), -math.inf, dtype=torch.float64, device=DEV)
    best_i = torch.full((B, kmax), -1, dtype=torch.int64, device=DEV)
    all_s, all_w = [], []
    for a0 in range(0, n, step):
        m = min(step, n - a0)
        deep = x["emb"][a0:a0 + m].double() @ h.T  # [m][B]
        if c["op"] == "noalloc":
            wide = x["wide"][a0:a0 + m, None].double()
        else:
            key = x["ad_key"][a0:a0 + m].long()
            key[key < 0] = x["n_keys"]
            wide = torch.zeros((m, B), dtype=torch.float64, device=DEV)
            for j in range(f):
                wide += wts[key[:, j]]
        s = deep + wide
        if c["op"] == "build":
            all_s.append(s[:, 0])
            all_w.append(wide[:, 0])
            continue
        s = s.T.contiguous()
        if x["filter"] is not None:
            for b in range(B):
                s[b] = _masked(s[b], x["filter"][b], a0)
        t, i = torch.topk(s, min(kmax, m), dim=1)
        t, i = torch.cat([best_s, t], 1), torch.cat([best_i, i + a0], 1)
        best_s, o = torch.topk(t, kmax, dim=1)
        best_i = torch.gather(i, 1, o)
    if c["op"] == "build":
        return {"scores": torch.cat(all_s), "wide": torch.cat(all_w), "info": None}
    best_i[torch.isinf(best_s)] = -1
    for b in range(B):
        best_s[b, ks[b]:] = -math.inf
        best_i[b, ks[b]:] = -1
    if c["op"] == "noalloc":
        best_s, best_i = best_s[0], best_i[0]
    ids = best_i.to(torch.int32)
    return {"ids": ids.cpu().numpy().view(np.uint32) if c["host"] else ids, "scores": best_s}
