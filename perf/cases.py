"""Timed cases of the search calls: what a retrieval service has the library do, from one query against a small corpus
to a batch of 256 against 8.8 million documents.

A case names a corpus shape, the form of the residual codes, the query batch and the search parameters.  The corpora
are synthetic stand-ins of the same kind as synth/corpus.py's (mixture means as centroids, tokens that pick a
component, residuals well inside the middle code buckets, queries from the same mixture), drawn directly in their
encoded form on the GPU so that the largest one takes well under a second.
"""
import math

import torch

from paper_2608_23553_b200.binding import Index

INT32_MIN = -(1 << 31)
CHUNK = 1 << 26                     # 32-bit words generated at a time


def _case(name, **kw):
    """Fills in the ordinary choices: 128-dimensional 2-bit codes, 32-token queries, 4 probes, pruning by centroid
    interaction, device buffers."""
    c = {"name": name, "mode": "ci", "host": False, "n_docs": 10_000, "len_kind": "uniform", "len_lo": 32, "len_hi": 96,
         "len_mid": 64, "n_centroids": 1_024, "skew": 1.0, "dim": 128, "nbits": 2, "batch": 1, "q_len": 32, "nprobe": 4, "n_prune": 256,
         "k": 10}
    c.update(kw)
    return c


TINY = {"n_docs": 10_000, "len_lo": 32, "len_hi": 96, "n_centroids": 1_024, "n_prune": 256, "k": 10}
MID = {"n_docs": 500_000, "len_lo": 40, "len_hi": 200, "n_centroids": 65_536, "n_prune": 1_024, "k": 10}
LARGE = {"n_docs": 8_800_000, "len_kind": "lognormal", "len_lo": 8, "len_hi": 180, "len_mid": 61, "n_centroids": 262_144,
         "n_prune": 4_096, "k": 100}
LONG = {"n_docs": 200_000, "len_kind": "fixed", "len_lo": 512, "len_hi": 512, "n_centroids": 32_768, "q_len": 64,
        "nprobe": 8, "n_prune": 2_048, "k": 50}


def listed():
    return [
        # one interactive query against a small private corpus: launches and latency
        _case("tiny_b1", **TINY),
        # one interactive query against half a million documents
        _case("mid_b1", **MID),
        # a throughput batch of the same corpus, with each of the library's pruning methods: every token of every
        # candidate; the retrieved tokens only; 1-bit codes; 1-bit codes with probes from the centroid graph
        _case("mid_b256", batch=256, **MID),
        _case("mid_partial_b256", mode="partial", batch=256, **MID),
        _case("mid_rabitq_b256", mode="rabitq", batch=256, **MID),
        _case("mid_graph_b64", mode="graph", batch=64, **MID),
        # passage retrieval at full size: one query from host memory and back, as a query server issues it ...
        _case("large_host_b1", host=True, **LARGE),
        # ... and the largest batch
        _case("large_b256", batch=256, **LARGE),
        # long documents, long queries
        _case("long_b64", batch=64, **LONG),
        # unpadded queries over 1-bit 96-dimensional codes, ragged documents, popular centroids, an odd batch
        _case("ragged_b37", n_docs=123_457, len_kind="lognormal", len_lo=1, len_hi=300, len_mid=70, n_centroids=16_411,
              skew=1.5, dim=96, nbits=1, batch=37, q_len=21, nprobe=6, n_prune=777, k=25),
        # a passage as the query (more than 64 tokens)
        _case("passage_query_b8", n_docs=200_000, len_lo=20, len_hi=180, n_centroids=32_768, batch=8, q_len=100, nprobe=4,
              n_prune=1_024, k=20),
        # recall first: many probes, deep pruning list and a long result, served through host buffers
        _case("deep_host_b16", host=True, n_docs=500_000, len_lo=40, len_hi=200, n_centroids=65_536, batch=16, nprobe=32,
              n_prune=16_384, k=1_000),
    ]


# ---------------------------------------------------------------------------------------------- sizes -------------
def _len_mean(c):
    """Mean document length of the case (log-normal lengths have the median len_mid and sigma 0.5)."""
    return c["len_mid"] * 1.12 if c["len_kind"] == "lognormal" else (c["len_lo"] + c["len_hi"]) / 2


def _candidate_share(c):
    """Expected share of the documents that own a token of a probed centroid."""
    probed = min(1.0, c["q_len"] * c["nprobe"] / c["n_centroids"])
    return 1.0 - (1.0 - probed) ** _len_mean(c)


def _capacity(c):
    """max_candidates: all documents for small corpora, else two fifths above the mean length of the probed lists."""
    if c["n_docs"] <= 1_000_000:
        return 0
    postings = c["q_len"] * c["nprobe"] * c["n_docs"] * _len_mean(c) / c["n_centroids"]
    return min(c["n_docs"], (int(postings * 1.4) // 1024 + 1) * 1024)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Corpora of 2 thousand to 2 million documents with 1 to 512 tokens each, 400 to 3,500 tokens per centroid,
    batches of 1 to 256, queries of 4 to 127 tokens (mostly the padded 32 and 64), every code form and pruning method."""
    n_docs = _log(rng, 2_000, 2_000_000)
    kind = rng.choice(["uniform", "lognormal", "fixed"])
    hi = rng.randint(16, 512 if n_docs < 250_000 else 200)
    lo = hi if kind == "fixed" else rng.randint(1, hi // 2)
    mode = rng.choice(["ci", "ci", "ci", "partial", "rabitq", "graph"])
    q_len = rng.choice([32, 32, 32, 64, rng.randint(4, 64), rng.randint(65, 127)])
    c = {"mode": mode, "host": mode == "ci" and rng.random() < 0.25, "n_docs": n_docs, "len_kind": kind, "len_lo": lo,
         "len_hi": hi, "len_mid": rng.randint(lo, hi // 2) if kind == "lognormal" else (lo + hi) // 2,
         "skew": rng.choice([1.0, 1.0, 1.5]) if n_docs <= 1_000_000 else 1.0, "dim": rng.choice([128, 128, 96, 64, 32]),
         "nbits": rng.choice([2, 2, 1]), "q_len": q_len}
    c["n_centroids"] = max(256, min(262_144, int(n_docs * _len_mean(c) / _log(rng, 400, 3_500))))
    if mode in ("rabitq", "graph"):
        c["q_len"] = q_len = min(q_len, 64)
    c["nprobe"] = min(_log(rng, 1, 32), c["n_centroids"])
    c["n_prune"] = min(16_384, max(16, _log(rng, 64, 16_384)))
    c["k"] = min(_log(rng, 1, 1_000), c["n_prune"])
    # the batch: as large as wanted while the scanned tokens, the score table and the workspace stay below those of
    # the largest listed case
    batch = _log(rng, 1, 256)
    scanned = n_docs * _candidate_share(c) * _len_mean(c) * max(q_len, 32) / 32
    table = c["n_centroids"] * q_len
    rows = (_capacity(c) or n_docs) * (q_len + 16 if mode != "ci" else 16) * 4
    late = c["n_prune"] * _len_mean(c) * q_len * c["dim"]
    c["batch"] = int(max(1, min(batch, 2e9 / scanned, 2e9 / table, 16e9 / rows, 4e11 / late)))
    return c


def work(case):
    """One pass: the centroids, posting lists, centroid ids and codes it has to look at, each byte once however many
    queries of the batch want it, and the products of the two contractions."""
    c = case
    B, nq, D, K, N = c["batch"], c["q_len"], c["dim"], c["n_centroids"], c["n_docs"]
    L = _len_mean(c)
    seen = 1.0 - (1.0 - min(1.0, nq * c["nprobe"] / K)) ** B             # share of the lists probed by the batch
    postings = N * L * seen
    cand = N * _candidate_share(c)                                       # candidates of one query
    cand_any = N * (1.0 - (1.0 - seen) ** L)                             # ... of any query of the batch
    kept = min(c["n_prune"], cand)
    kept_any = min(N, B * kept)
    one_bit = c["mode"] in ("rabitq", "graph")
    code = D // 8 + 4 if one_bit else D * c["nbits"] // 8 + 4            # code and factor, or code and centroid id
    retrieved = N * L * min(1.0, nq * c["nprobe"] / K)                   # tokens of one query's lists
    io = B * (4 * nq * D + 8 * c["k"])
    if c["mode"] == "ci":
        nbytes = 4 * K * D + 4 * postings + cand_any * (4 * L + 8) + kept_any * L * (code - 4)
        flops = 2 * B * nq * (K * D + kept * L * D) + B * cand * L * nq
    else:
        centroids = 0.1 * K if c["mode"] == "graph" else K
        nbytes = 4 * centroids * D + postings * (8 + code) + kept_any * L * code
        flops = 2 * B * nq * D * (centroids + kept * L) + 2 * B * retrieved * D
    return {"bytes": int(nbytes + io), "flops": int(flops)}


def tolerance(case):
    """The 1-bit pipeline's results are defined bit for bit.  Otherwise the scores are 32-bit sums, and documents whose
    scores agree to rounding may come in either order."""
    if case["mode"] in ("rabitq", "graph"):
        return "exact"
    return {"rel": 1e-5, "max": 1e-4, "differ": 0.005}


# ---------------------------------------------------------------------------------------------- inputs ------------
def _doc_lengths(c, g):
    n, lo, hi = c["n_docs"], c["len_lo"], c["len_hi"]
    if c["len_kind"] == "fixed":
        return torch.full((n,), lo, dtype=torch.int32, device="cuda")
    if c["len_kind"] == "uniform":
        return torch.randint(lo, hi + 1, (n,), generator=g, dtype=torch.int32, device="cuda")
    x = c["len_mid"] * torch.exp(0.5 * torch.randn(n, generator=g, device="cuda"))
    return x.round_().clamp_(lo, hi).to(torch.int32)


def _components(c, n, g):
    """n mixture components: uniform, or (skew > 1) with popular ones."""
    K = c["n_centroids"]
    if c["skew"] == 1.0:
        return torch.randint(0, K, (n,), generator=g, dtype=torch.int32, device="cuda")
    u = torch.rand(n, generator=g, device="cuda")
    return (u.pow_(c["skew"]) * K).to(torch.int32).clamp_(max=K - 1)


def _words(n, g):
    return torch.empty(n, dtype=torch.int32, device="cuda").random_(INT32_MIN, 1 << 31, generator=g)


def _codes(c, T, g):
    """[T, dim * nbits / 8] packed residual codes: signs for one bit, the two middle buckets for two."""
    words = torch.empty(T * (c["dim"] * c["nbits"] // 32), dtype=torch.int32, device="cuda")
    for i in range(0, words.numel(), CHUNK):
        w = _words(min(CHUNK, words.numel() - i), g)
        if c["nbits"] == 2:                                              # 01 or 10 in every pair of bits
            w = (w & 0x55555555) | ((~w & 0x55555555) << 1)
        words[i:i + CHUNK] = w
    return words.view(torch.uint8).view(T, -1)


def _one_bit_codes(c, means, cids, g):
    """Rotation, sign bits of the rotated tokens (those of the rotated centroid with about one in eight flipped by the
    token's own part) and the tokens' factors."""
    K, D = means.shape
    rot = torch.linalg.qr(torch.randn(D, D, generator=g, device="cuda", dtype=torch.float64))[0].to(torch.float32)
    shifts = torch.arange(8, device="cuda", dtype=torch.int32)
    sign = ((means @ rot.t() > 0).to(torch.int32).view(K, D // 8, 8) << shifts).sum(dim=2).to(torch.uint8)
    sign = sign.view(torch.int32)                                        # [K, D / 32]
    T, W = cids.numel(), D // 32
    bits = torch.empty(T, W, dtype=torch.int32, device="cuda")
    step = CHUNK // W
    for i in range(0, T, step):
        n = min(step, T - i)
        flip = _words(n * W, g) & _words(n * W, g) & _words(n * W, g)
        bits[i:i + n] = sign[cids[i:i + n].long()] ^ flip.view(n, W)
    inv = 1.2533 * (1.0 + 0.05 * torch.randn(T, generator=g, device="cuda").clamp_(-3, 3))
    return rot.contiguous(), bits.view(torch.uint8).view(T, D // 8), inv


def prepare(case, seed):
    c = case
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    means = torch.randn(c["n_centroids"], c["dim"], generator=g, device="cuda")
    centroids = means / means.norm(dim=1, keepdim=True)
    doclens = _doc_lengths(c, g)
    T = int(doclens.sum(dtype=torch.int64))
    cids = _components(c, T, g)
    codes = _codes(c, T, g)
    index = Index(centroids, cids, codes, doclens, c["nbits"])
    if c["mode"] == "partial":
        index.enable_partial()
    elif c["mode"] in ("rabitq", "graph"):
        index.attach_rabitq(*_one_bit_codes(c, means, cids, g))
        if c["mode"] == "graph":
            index.build_graph(min(32, c["n_centroids"] - 1))
    x = means[_components(c, c["batch"] * c["q_len"], g).long()]
    x = x + 0.3 * torch.randn(x.shape, generator=g, device="cuda")
    queries = (x / x.norm(dim=1, keepdim=True)).view(c["batch"], c["q_len"], c["dim"]).contiguous()
    return {"index": index, "queries": queries.cpu().pin_memory() if c["host"] else queries, "host": c["host"],
            "args": (c["nprobe"], c["n_prune"], c["k"], _capacity(c)),
            "options": {"partial": {"partial": True}, "rabitq": {"rabitq": True},
                        "graph": {"rabitq": True, "graph": (32, min(256, c["n_centroids"]), 1 << 30)}}.get(c["mode"], {})}


def run(state):
    """One search call: (ids [batch, k], scores [batch, k])."""
    index = state["index"]
    if state["host"]:
        return index.search_host(state["queries"], *state["args"])
    return index.search(state["queries"], *state["args"], **state["options"])
