"""The measured work of this framework: what a deduplication program has it do.

A program builds an IVF index of its embeddings once (``build_layout``, and
``build_rq_layout`` for 7-bit codes), keeps it in device memory and searches
batches of records against it: single records as they arrive, small and
medium batches, and whole-corpus self-joins.  Each case below is one such
call through the public Python entry points; sizes, thresholds, windows and k
are those of this repository's configurations, tests and benchmark, or odd
neighbours of them.

Inputs are clustered unit-norm embeddings with planted near-duplicate
families: centroids in groups of eight neighbours (cosine about 0.94), rows
around them, skewed partition sizes, every row assigned to the nearest
centroid of its group.  A family's copies lie either well above the threshold
or well below it, so that no output hinges on the last bit of a similarity.
Queries are rows of the corpus (self-join), each excluded from its own result
by its id.
"""
import math

import torch

import paper_2608_03199_gb300 as sieve

DEV = "cuda"
GROUP = 8          # neighbouring centroids per group
BITS = 7           # code width of the quantized search


def listed():
    return [
        # one record checked against the index as it arrives: pure latency
        dict(name="one_query", op="search", n=1_000_000, d=256, nlist=1024, dup=0.08, heavy=True,
             nq=1, tau=0.90, k=10, nprobe=64, W=8, lookahead=True),
        # a small batch on a small index, every size odd
        dict(name="small_odd", op="search", n=50_021, d=100, nlist=149, dup=0.05, heavy=False,
             nq=1_003, tau=0.90, k=7, nprobe=24, W=4, lookahead=True),
        # an ordinary batch from host memory, results back on the host
        dict(name="host_10k", op="host", n=1_000_000, d=256, nlist=1024, dup=0.08, heavy=True,
             nq=10_007, tau=0.90, k=10, nprobe=64, W=8, lookahead=True),
        # a tenth of a 1M corpus joined against it, the stopping rule on
        dict(name="join_1m", op="search", n=1_000_000, d=256, nlist=1024, dup=0.08, heavy=True,
             nq=100_000, tau=0.90, k=10, nprobe=64, W=8, lookahead=True),
        # the same with fixed probing (the exhaustive reference of the rule,
        # and what calibration runs on its sample)
        dict(name="fixed_1m", op="search", n=1_000_000, d=256, nlist=1024, dup=0.08, heavy=True,
             nq=100_000, tau=0.90, k=10, nprobe=64, W=64, lookahead=True),
        # the same over 7-bit codes
        dict(name="codes_1m", op="rq", n=1_000_000, d=256, nlist=1024, dup=0.08, heavy=True,
             nq=99_991, tau=0.90, k=10, nprobe=64, W=8, lookahead=True),
        # a large batch against a 10M corpus
        dict(name="join_10m", op="search", n=10_000_000, d=256, nlist=8192, dup=0.03, heavy=False,
             nq=1_000_000, tau=0.95, k=10, nprobe=128, W=8, lookahead=True),
        # wide rows: no tensor-core layout is built above d = 256 by default
        dict(name="wide_512", op="search", n=5_000_000, d=512, nlist=16384, dup=0.05, heavy=True,
             nq=200_000, tau=0.92, k=10, nprobe=128, W=8, lookahead=True),
        # the largest: a million records, 65,536 partitions of narrow rows
        dict(name="join_32m", op="search", n=32_000_000, d=96, nlist=65536, dup=0.04, heavy=False,
             nq=1_000_000, tau=0.90, k=10, nprobe=256, W=8, lookahead=True),
        # the centroid ranking alone (kept by programs that search the same
        # batch with several settings)
        dict(name="rank_65k", op="rank", n=262_144, d=96, nlist=65536, dup=0.0, heavy=False,
             nq=100_000, tau=0.90, k=10, nprobe=256, W=8, lookahead=True),
        # independent index shards searched one after the other and merged
        dict(name="shards_8", op="shards", n=4_000_000, d=96, nlist=12_000, dup=0.04, heavy=False,
             nq=100_000, tau=0.90, k=10, nprobe=90, W=8, lookahead=True, shards=8),
        # building the index from rows and their partitions
        dict(name="build_1m", op="build", n=1_000_000, d=256, nlist=1024, dup=0.08, heavy=True,
             nq=0, tau=0.90, k=10, nprobe=64, W=8, lookahead=True),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["search"] * 6 + ["host", "rq", "rank", "shards", "build"])
    d = rng.choice([32, 64, 96, 100, 128, 192, 200, 256] + ([] if op in ("rq", "shards") else [384, 512]))
    nlist = _spread(rng, 64, 65_536 if op == "rank" else 16_384 if op == "search" else 4_096)
    n = max(20_000, min(4_000_000, nlist * (4 if op == "rank" else _spread(rng, 100, 1_500))))
    nq = min(n, _spread(rng, 1, 200_000))
    nprobe = min(nlist, _spread(rng, 8, 256))
    W = min(nprobe, rng.choice([2, 4, 8, 8, 8, 16, 256]))
    shards = 0
    if op == "shards":
        shards = rng.choice([2, 4, 8])
        nlist = max(64, nlist // shards) * shards
        nprobe = min(nprobe, nlist // shards)
        W = min(W, nprobe)
    # no drawn batch costs more than the largest listed one
    per_query = 2.0 * d * (nlist + (0 if op == "rank" else max(1, shards) * W * n / nlist))
    nq = max(1, min(nq, int(2e12 / per_query)))
    c = dict(op=op, n=n, d=d, nlist=nlist, dup=rng.choice([0.02, 0.05, 0.1]), heavy=rng.random() < 0.5,
             nq=nq, tau=rng.choice([0.90, 0.92, 0.95]), k=rng.choice([1, 5, 10, 10, 10, 20, 50]),
             nprobe=nprobe, W=W, lookahead=op == "shards" or rng.random() < 0.9)
    if shards:
        c["shards"] = shards
    return c


# ---------------------------------------------------------------------------
# inputs
def _unit(x):
    return x / x.norm(dim=1, keepdim=True)


def _corpus(case, seed):
    """Rows [n][d], their partitions [n], centroids [nlist][d], query rows [nq]."""
    n, d, nlist, tau = case["n"], case["d"], case["nlist"], case["tau"]
    g = torch.Generator(DEV).manual_seed(seed)

    def randn(*shape):
        return torch.randn(*shape, generator=g, device=DEV)

    base = _unit(randn(-(-nlist // GROUP), d))
    cent = _unit(base.repeat_interleave(GROUP, 0)[:nlist] + 0.25 * randn(nlist, d) / math.sqrt(d))
    sigma = 0.7 + 0.6 * torch.rand(nlist, generator=g, device=DEV)
    cum = torch.exp(0.6 * randn(nlist)).double().cumsum(0)
    ncopy = int(case["dup"] * n)
    nbase = n - ncopy
    comp = torch.searchsorted(cum, cum[-1] * torch.rand(nbase, generator=g, device=DEV, dtype=torch.float64))
    comp.clamp_(max=nlist - 1)
    step = max(1, (1 << 28) // (GROUP * d))
    X = torch.empty(n, d, device=DEV)
    for s in range(0, nbase, step):
        c = comp[s:s + step]
        X[s:min(s + step, nbase)] = _unit(cent[c] + sigma[c, None] * randn(len(c), d) / math.sqrt(d))
    if ncopy:
        # the first rows are parents; family sizes 1-5, or heavy-tailed up to 200
        u = torch.rand(ncopy, generator=g, device=DEV, dtype=torch.float64)
        size = (1 / u.clamp_min(1e-6)).long().clamp_(max=200) if case["heavy"] else 1 + (5 * u).long().clamp_(max=4)
        parent = torch.searchsorted(size.cumsum(0), torch.arange(ncopy, device=DEV), right=True) % nbase
        near = torch.rand(ncopy, generator=g, device=DEV)[parent % ncopy] < 0.6   # by family
        for s in range(0, ncopy, step):
            e = min(s + step, ncopy)
            p = X[parent[s:e]]
            v = randn(e - s, d)
            v = _unit(v - (v * p).sum(1, keepdim=True) * p)
            r = torch.rand(e - s, generator=g, device=DEV)
            # cosine to the parent, in units of 1 - tau: 0.01-0.2 or 1.6-2.2
            cos = 1 - (1 - tau) * torch.where(near[s:e], 0.01 + 0.19 * r, 1.6 + 0.6 * r)
            X[nbase + s:nbase + e] = _unit(cos[:, None] * p + (1 - cos * cos).sqrt()[:, None] * v)
        comp = torch.cat([comp, comp[parent]])
    perm = torch.randperm(n, generator=g, device=DEV)
    X, comp = X[perm], comp[perm]
    assign = torch.empty(n, dtype=torch.int32, device=DEV)
    for s in range(0, n, step):
        near_c = (comp[s:s + step, None] // GROUP * GROUP
                  + torch.arange(GROUP, device=DEV)).clamp_(max=nlist - 1)
        x = X[s:s + step]
        best = torch.bmm(cent[near_c], x[:, :, None])[:, :, 0].argmax(1, keepdim=True)
        assign[s:s + step] = near_c.gather(1, best)[:, 0].int()
    # centroid ids in random order (within a shard): neighbours are not adjacent
    shard = torch.arange(nlist, device=DEV) // (nlist // max(1, case.get("shards", 0)))
    slot = (torch.rand(nlist, generator=g, device=DEV) + shard).argsort().argsort()
    assign = slot[assign.long()].int()
    cent = torch.empty_like(cent).index_copy_(0, slot, cent)
    if case["op"] == "build":   # every seed the same partition sizes, so outputs of one shape
        w = torch.exp(0.6 * torch.randn(nlist, generator=torch.Generator().manual_seed(7)))
        size = (n * w / w.sum()).long()
        size[0] += n - size.sum()
        assign = torch.repeat_interleave(torch.arange(nlist), size).int().to(DEV)[perm]
    if case["nq"] >= 64 or not ncopy:
        rows = torch.randperm(n, generator=g, device=DEV)[:case["nq"]]
    else:   # a few records: ones that have something to find
        copies = torch.empty_like(perm).index_copy_(0, perm, torch.arange(n, device=DEV))[nbase:][near]
        rows = copies[torch.randperm(len(copies), generator=g, device=DEV)[:case["nq"]]]
    return X, assign, cent, rows


def _rotation(d):
    """A seeded random orthogonal matrix (float64)."""
    g = torch.Generator("cpu").manual_seed(7)
    q, r = torch.linalg.qr(torch.randn(d, d, generator=g, dtype=torch.float64))
    return (q * torch.sign(torch.diagonal(r))).contiguous().to(DEV)


def _shard_rows(case, assign):
    """Per shard: its rows and its centroids (contiguous ranges of partitions)."""
    per = case["nlist"] // case["shards"]
    which = assign // per
    return per, [(which == s).nonzero()[:, 0] for s in range(case["shards"])]


def prepare(case, seed):
    X, assign, cent, rows = _corpus(case, seed)
    st = dict(case=case)
    if case["op"] == "build":
        blocks = int(((torch.bincount(assign, minlength=case["nlist"]) + 127) // 128).sum())
        st.update(X=X, assign=assign, cent=cent, blocks=blocks)
        return st
    st.update(Q=X[rows], qids=rows)
    if case["op"] == "host":
        nq, k = case["nq"], case["k"]
        st["Q"] = st["Q"].cpu().pin_memory()
        st["qids"] = rows.cpu().pin_memory()
        st["out"] = (torch.empty(nq, k, dtype=torch.int64).pin_memory(), torch.empty(nq, k).pin_memory(),
                     torch.empty(nq, dtype=torch.int32).pin_memory(),
                     torch.empty(nq, dtype=torch.int32).pin_memory())
    if case["op"] == "shards":
        st["index"] = []
        per, parts = _shard_rows(case, assign)
        for s, r in enumerate(parts):
            ix = sieve.build_layout(X[r], assign[r] - s * per, per, cent[s * per:(s + 1) * per].contiguous())
            ix.ids = r[ix.ids]
            st["index"].append(ix)
        return st
    st["index"] = sieve.build_layout(X, assign, case["nlist"], cent)
    if case["op"] == "rq":
        st["rq"] = sieve.build_rq_layout(st["index"], _rotation(case["d"]), BITS)
    return st


# ---------------------------------------------------------------------------
# one pass
def run(st):
    c = st["case"]
    if c["op"] == "build":
        ix = sieve.build_layout(st["X"], st["assign"], c["nlist"], st["cent"])
        out = dict(vectors=ix.vectors, ids=ix.ids, offsets=ix.list_offsets)
        if ix.tc_rows is not None:   # the blocks and a norm for each: what is written of the buffer
            used = st["blocks"] * (-(-c["d"] // 64) * 32768 + 4)
            out.update(rows=ix.tc_rows[:used], blocks=ix.tc_row_blocks, centroids=ix.tc_centroids)
        return out
    if c["op"] == "rank":
        order, scores = sieve.rank_partitions(st["index"], st["Q"], c["nprobe"], return_scores=True)
        return dict(order=order, scores=scores)
    args = (st["Q"], c["tau"], c["k"], c["nprobe"], c["W"])
    if c["op"] == "host":
        out = sieve.search_host(st["index"], *args, lookahead=c["lookahead"], query_ids_host=st["qids"],
                                out=st["out"])
    elif c["op"] == "rq":
        out = sieve.rq_search(st["index"], st["rq"], *args, lookahead=c["lookahead"], query_ids=st["qids"])
    elif c["op"] == "shards":
        out = sieve.sharded_search(st["index"], *args, lookahead=c["lookahead"], query_ids=st["qids"])
    else:
        out = sieve.search(st["index"], *args, lookahead=c["lookahead"], query_ids=st["qids"])
    return dict(zip(("ids", "scores", "count", "probes", "shard_probes"), out))


def work(case):
    n, d, nlist, nq, k = (case[x] for x in ("n", "d", "nlist", "nq", "k"))
    if case["op"] == "build":   # rows, partitions and centroids in; rows, ids and the split copy out
        copies = 4 if d <= sieve.TC_BULK_MAX_D else 2
        return {"bytes": n * (4 * d * (copies - 1) + 12) + nlist * (4 * d * (copies - 1) + 8), "flops": 2 * n * d}
    queries = nq * (4 * d + 8)
    rank = 2.0 * d * nq * nlist
    if case["op"] == "rank":
        return {"bytes": nq * 4 * d + nlist * 4 * d + nq * case["nprobe"] * 8, "flops": rank}
    probes = min(case["W"], case["nprobe"]) * max(1, case.get("shards", 0))
    per = n / nlist
    row = d + 4 if case["op"] == "rq" else 4 * d
    rows = min(nlist, nq * probes) * per * row
    flops = rank + 2.0 * d * nq * probes * per + (2.0 * d * d * nq if case["op"] == "rq" else 0)
    return {"bytes": queries + nlist * 4 * d + rows + nq * (12 * k + 8), "flops": flops}


def tolerance(case):
    if case["op"] == "build":
        return "exact"
    # against exact() the scores are off by up to 3.4e-7 (ranking, d = 96), 1.2e-6
    # (codes, d = 256) and 3.3e-6 (three fp16 products, d = 512), growing with d,
    # and near-ties change places in up to 2.5e-4 of the ids: four times that
    return {"rel": 2.5e-8 * case["d"], "max": 5e-8 * case["d"], "differ": 1e-3}


# ---------------------------------------------------------------------------
# the same in 64 bits, with torch alone
def _rank64(Q, cent, nprobe):
    Cd = cent.double()
    order, scores = [], []
    for q in Q.split(max(1, (1 << 28) // cent.shape[0])):
        s, o = (q.double() @ Cd.T).topk(nprobe, dim=1)
        order.append(o)
        scores.append(s)
    return torch.cat(order), torch.cat(scores)


def _pair_scores(case, X, assign, cent, Q, q, r, P):
    """64-bit similarity of queries q and rows r, or its estimate from codes."""
    out = torch.empty(len(q), dtype=torch.float64, device=DEV)
    if P is not None:
        rows, at = r.unique(return_inverse=True)
        c = cent[assign[rows].long()].double()
        res = X[rows].double() - c
        norm = res.norm(dim=1)
        o = (res / norm.clamp_min(1e-300)[:, None]) @ P
        top = float((1 << BITS) - 1)
        delta = 2 * o.abs().amax(1, keepdim=True) / top
        u = (o / delta + top / 2).round().clamp(0, top) - top / 2
        f = (norm / (u * o).sum(1)).float().double()
        Qr = Q.double() @ P
    for s in range(0, len(q), 1 << 18):
        a, b = q[s:s + (1 << 18)], r[s:s + (1 << 18)]
        if P is None:
            out[s:s + (1 << 18)] = (Q[a].double() * X[b].double()).sum(1)
        else:
            i = at[s:s + (1 << 18)]
            out[s:s + (1 << 18)] = (Q[a].double() * c[i]).sum(1) + f[i] * (u[i] * Qr[a]).sum(1)
    return out


def _visit64(case, X, assign, cent, Q, qids, ids, P=None):
    """The qualifying (query, id, score) of the searched partitions, and the probes."""
    nq, W = Q.shape[0], case["W"]
    nprobe, tau = case["nprobe"], case["tau"]
    order, _ = _rank64(Q, cent, nprobe)
    by_part = assign.sort(stable=True).indices
    off = [0] + torch.bincount(assign, minlength=cent.shape[0]).cumsum(0).tolist()
    stop = torch.full((nq,), min(W, nprobe), dtype=torch.int64, device=DEV)
    done = torch.zeros_like(stop)
    ranks = torch.arange(nprobe, device=DEV)
    found = []
    slack = 1e-3 if P is None else 0.05
    while True:
        q, r = ((ranks[None] >= done[:, None]) & (ranks[None] < stop[:, None])).nonzero(as_tuple=True)
        if not len(q):
            break
        done = stop.clone()
        p, at = order[q, r].sort()
        q, r = q[at], r[at]
        part, cnt = p.unique_consecutive(return_counts=True)
        pairs, i = [], 0
        for a, m in zip(part.tolist(), cnt.tolist()):
            rows = by_part[off[a]:off[a + 1]]
            x, y = (Q[q[i:i + m]] @ X[rows].T >= tau - slack).nonzero(as_tuple=True)
            pairs.append((x + i, rows[y]))
            i += m
        item, row = (torch.cat(v) for v in zip(*pairs))
        s = _pair_scores(case, X, assign, cent, Q, q[item], row, P)
        keep = (s >= tau) & (ids[row] != qids[q[item]])
        item, row, s = item[keep], row[keep], s[keep]
        found.append((q[item], ids[row], s))
        stop.scatter_reduce_(0, q[item], (r[item] + 1 + W).clamp(max=nprobe), "amax")
    return [torch.cat(v) for v in zip(*found)], stop


def _top64(found, nq, k):
    q, i, s = found
    # by query, then score (best first), then id: stable sorts, last key first
    for key in (lambda: i, lambda: -s, lambda: q):
        at = key().sort(stable=True).indices
        q, i, s = q[at], i[at], s[at]
    total = torch.bincount(q, minlength=nq)
    place = torch.arange(len(q), device=DEV) - (total.cumsum(0) - total)[q]
    in_k = place < k
    ids = torch.full((nq, k), -1, dtype=torch.int64, device=DEV)
    scores = torch.full((nq, k), -math.inf, dtype=torch.float64, device=DEV)
    ids[q[in_k], place[in_k]] = i[in_k]
    scores[q[in_k], place[in_k]] = s[in_k]
    return ids, scores, total.clamp(max=k).int()


def exact(case, seed):
    if case["op"] == "build" or (case["op"] != "rank" and (case["nlist"] > 9000 * max(1, case.get("shards", 0)))):
        return None   # bytes and copies; or a Python loop over too many partitions
    X, assign, cent, rows = _corpus(case, seed)
    Q = X[rows]
    if case["op"] == "rank":
        order, scores = _rank64(Q, cent, case["nprobe"])
        return dict(order=order.int(), scores=scores)
    if case["op"] == "shards":
        per, parts = _shard_rows(case, assign)
        found, probes = [], []
        for s, r in enumerate(parts):
            f, p = _visit64(case, X[r], assign[r] - s * per, cent[s * per:(s + 1) * per], Q, rows, r)
            found.append(f)
            probes.append(p)
        ids, scores, count = _top64([torch.cat(v) for v in zip(*found)], case["nq"], case["k"])
        per_shard = torch.stack(probes, 1).int()
        return dict(ids=ids, scores=scores, count=count, probes=per_shard.sum(1).int(), shard_probes=per_shard)
    P = _rotation(case["d"]) if case["op"] == "rq" else None
    found, probes = _visit64(case, X, assign, cent, Q, rows, torch.arange(case["n"], device=DEV), P)
    ids, scores, count = _top64(found, case["nq"], case["k"])
    return dict(ids=ids, scores=scores, count=count, probes=probes.int())
