"""The work that users of this framework have it do, as cases to be timed: index builds,
batched and single searches, uneven batches, and the brute-force K-NN behind ground truth
and graph building, each through the package's public calls.

Data follow the recipes of `workloads` (latent mixtures shaped like SIFT, GloVe, DEEP and
GIST), drawn on the GPU so that an input of a million rows takes a second.  Graphs are
relative-neighbourhood pruned K-NN graphs over each point's own and nearest clusters, with
reverse edges, plus long links among a random sample of the nodes, from whose most central
one a search starts.
"""
import math

import torch

import paper_2402_11354_gb300 as peos

# Shape and statistics of each recipe: d, out-degree R, code blocks L, points per cluster,
# latent dimension and spread of the mixture (as in workloads.CONFIGS), and the clusters
# around a point among which its graph neighbours are looked for.
RECIPES = {
    "tiny": dict(d=128, R=32, L=8, per=200, latent=128, spread=0.3, reach=8),
    "sift": dict(d=128, R=32, L=8, per=1000, latent=16, spread=0.5, reach=24),
    "sift-hard": dict(d=128, R=32, L=8, per=1000, latent=32, spread=2.0, reach=64),
    "glove": dict(d=100, R=48, L=10, per=600, latent=20, spread=0.5, reach=32),
    "deep": dict(d=96, R=32, L=8, per=1000, latent=16, spread=0.5, reach=24),
    "gist": dict(d=960, R=32, L=24, per=200, latent=24, spread=0.5, reach=64),
}
M = 16           # random vectors per code block in every configuration
PROJ_SEED = 3001  # the index's own random vectors: part of its definition, not of the inputs


def listed():
    return [
        # one interactive query from host memory: latency of a single call
        dict(name="host-one", kind="host", recipe="sift", n=200_000, nq=1, k=10, ef=64, routing=1),
        # the small configuration: 100 queries, entry nodes from the upper layers, then the search
        dict(name="hier-100", kind="hier", recipe="tiny", n=10_000, nq=100, k=10, ef=16, routing=1),
        # the headline: 10,000 queries a call on a million SIFT-shaped rows at recall@10 of 0.95
        dict(name="sift-1m", kind="search", recipe="sift", n=1_000_000, nq=10_000, k=10, ef=18, routing=1),
        # the same call without the routing test
        dict(name="sift-1m-plain", kind="search", recipe="sift", n=1_000_000, nq=10_000, k=10, ef=16, routing=0),
        # out-degree 48, unit vectors, 8-bit rows with the exact re-rank of every list
        dict(name="glove-e4m3", kind="search", recipe="glove", n=300_000, nq=10_000, k=10, ef=18, routing=1,
             storage="e4m3", rerank=True),
        # long rows
        dict(name="gist", kind="search", recipe="gist", n=200_000, nq=10_000, k=10, ef=42, routing=1),
        # long searches, two nodes an iteration
        dict(name="hard-beam2", kind="search", recipe="sift-hard", n=300_000, nq=10_000, k=10, ef=144, routing=1,
             beam=2),
        # uneven k and efs in one launch, BF16 rows, exact re-rank, the caller's workspace
        dict(name="batch-deep-bf16", kind="batch", recipe="deep", n=500_000, nq=20_000, k=100, ef=512, routing=1,
             storage="bf16", rerank=True),
        # index-time codes of a million rows, and of long rows
        dict(name="build-sift-1m", kind="build", recipe="sift", n=1_000_000),
        dict(name="build-gist", kind="build", recipe="gist", n=50_000),
        # ground truth: exact FP32 K-NN of float rows, and the tensor-core K-NN of a million rows
        dict(name="knn-exact-glove", kind="knn", recipe="glove", n=300_000, nq=2_000, k=100),
        dict(name="knn-tensor-1m", kind="knn_tensor", recipe="sift", n=1_000_000, nq=10_000, k=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "host", "hier", "batch", "build", "build", "knn", "knn_tensor"])
    if kind == "knn":
        # d = 96..960, with float and integer rows
        return dict(kind=kind, recipe=rng.choice(["sift", "glove", "deep", "gist"]), n=_log_int(rng, 5_000, 200_000),
                    nq=_log_int(rng, 1, 2_000), k=_log_int(rng, 1, 128))
    if kind == "knn_tensor":
        # integer rows below 256 are exact in BF16: the ranking has one answer
        return dict(kind=kind, recipe="sift", n=_log_int(rng, 5_000, 800_000), nq=_log_int(rng, 100, 20_000),
                    k=_log_int(rng, 1, 65))
    recipe = rng.choice(["sift", "sift", "glove", "deep", "gist", "sift-hard"])
    n = _log_int(rng, 10_000, 50_000 if recipe == "gist" else 250_000)
    if kind == "build":
        # FP32 edge scalars, or the compact 16/8-bit form
        return dict(kind=kind, recipe=recipe, n=n, scalar_bits=rng.choice([32, 32, 16, 8]))
    case = dict(kind=kind, recipe=recipe, n=n, k=rng.choice([1, 10, 10, 50]), routing=rng.choice([1, 1, 1, 0]))
    case["ef"] = max(case["k"], _log_int(rng, 10, 256))
    case["nq"] = _log_int(rng, 1, 200 if kind == "host" else 10_000)
    if kind in ("search", "batch"):
        case["storage"] = rng.choice(["f32", "f32", "bf16", "e4m3"])
        case["rerank"] = case["storage"] != "f32"
        case["beam"] = rng.choice([1, 1, 1, 2, 4])
    return case


# ------------------------------------------------------------------------------- data
def _points(recipe, n, gen):
    """n rows of the recipe in clusters of equal size: rows [clusters, per, d] (the last
    places surplus), and a function that draws more rows of the same mixture."""
    r = RECIPES[recipe]
    dev, d, lat = "cuda", r["d"], r["latent"]
    nc = max(1, round(n / r["per"]))
    per = -(-n // nc)

    def normal(*shape):
        return torch.randn(*shape, device=dev, generator=gen)

    centres = normal(nc, lat)
    image = None if recipe == "tiny" else normal(lat, d) / math.sqrt(lat)
    scales = torch.exp(0.75 * normal(d)) if recipe == "glove" else None

    def rows(labels):
        z = centres[labels] + r["spread"] * normal(len(labels), lat)
        if image is None:
            return z
        y = z @ image + 0.15 * normal(len(labels), d)
        if recipe in ("sift", "sift-hard"):
            return torch.round((48.0 * (y - 0.1).clamp_min(0.0)).clamp_max(255.0))
        if recipe == "gist":
            return (0.1 * (y - 0.1).clamp_min(0.0)).clamp(0.0, 1.0)
        if scales is not None:
            y = y * scales
        return y / y.norm(dim=1, keepdim=True)

    base = rows(torch.arange(nc, device=dev).repeat_interleave(per)).view(nc, per, d)

    def more(count):
        return rows(torch.randint(nc, (count,), device=dev, generator=gen)).contiguous()

    return base, more


def _prune(X, cand_d, cand_i, R, block=16384):
    """Relative-neighbourhood pruning of sorted candidate rows: c stays unless a kept s has
    d(s, c) < d(x, c).  Returns a mask over the candidates with at most R set in a row."""
    kept = torch.zeros_like(cand_i, dtype=torch.bool)
    block = max(1, block * 128 // X.shape[1])
    for s in range(0, len(cand_i), block):
        ci, cd = cand_i[s:s + block], cand_d[s:s + block]
        V = X[ci.clamp_min(0)]
        sq = (V * V).sum(-1)
        near = (sq.unsqueeze(2) + sq.unsqueeze(1) - 2.0 * torch.bmm(V, V.transpose(1, 2))) < cd.unsqueeze(1)
        ok = (ci >= 0) & torch.isfinite(cd)
        acc = torch.zeros_like(ok)
        for c in range(ci.shape[1]):
            acc[:, c] = ok[:, c] & ~(acc[:, :c] & near[:, :c, c]).any(1)
        acc &= torch.cumsum(acc.int(), 1) <= R
        kept[s:s + block] = acc
    return kept


def _union(n, R, owner, target, dist):
    """Each owner's R nearest of its own and its reversed edges, [n, R] ids (-1 = empty)."""
    o, t = torch.cat([owner, target]), torch.cat([target, owner])
    w = torch.cat([dist, dist])
    order = torch.argsort(o * n + t)
    o, t, w = o[order], t[order], w[order]
    first = torch.ones_like(o, dtype=torch.bool)
    first[1:] = (o[1:] != o[:-1]) | (t[1:] != t[:-1])
    o, t, w = o[first], t[first], w[first]
    order = torch.argsort(o * (1 << 32) + w.clamp_min(0.0).view(torch.int32).long(), stable=True)
    o, t = o[order], t[order]
    count = torch.bincount(o, minlength=n)
    rank = torch.arange(len(o), device=o.device) - (torch.cumsum(count, 0) - count)[o]
    fit = rank < R
    nbrs = torch.full((n, R), -1, dtype=torch.int32, device=o.device)
    nbrs[o[fit], rank[fit]] = t[fit].int()
    return nbrs


def _layer(X, R):
    """Pruned exact K-NN graph of a few thousand rows, local ids [len(X), R]."""
    n = len(X)
    D = torch.cdist(X, X, compute_mode="use_mm_for_euclid_dist").square()
    D.fill_diagonal_(float("inf"))
    w, t = torch.topk(D, min(2 * R, n - 1), largest=False)
    kept = _prune(X, w, t, R)
    owner = torch.arange(n, device=X.device).unsqueeze(1).expand_as(t)
    return _union(n, R, owner[kept], t[kept], w[kept])


def _graph(recipe, n, gen):
    """(X [n, d], nbrs [n, R] int32, entry, more): rows in random order and their graph."""
    base, more = _points(recipe, n, gen)
    nc, per, d = base.shape
    R, Kc = RECIPES[recipe]["R"], 64
    flat = base.view(-1, d)
    ids = torch.randperm(nc * per, device="cuda", generator=gen)  # place -> id, ids >= n are surplus
    X = torch.empty(n, d, device="cuda")
    real = ids < n
    X[ids[real]] = flat[real]
    sq = (flat * flat).sum(1)
    mean = base.mean(1)
    P = min(RECIPES[recipe]["reach"], nc)
    near = torch.cdist(mean, mean)
    near.fill_diagonal_(-1.0)
    near = torch.topk(near, P, largest=False).indices  # the cluster itself first
    own, tgt, dst = [], [], []
    step = max(1, (1 << 29) // (4 * per * per * P))
    places = torch.arange(nc * per, device="cuda").view(nc, per)
    for c in range(0, nc, step):
        pl = places[near[c:c + step]].reshape(-1, P * per)
        D = torch.baddbmm(sq[pl].unsqueeze(1), base[c:c + step], flat[pl].transpose(1, 2), alpha=-2.0)
        D += sq.view(nc, per)[c:c + step].unsqueeze(2)
        D.masked_fill_(~real[pl].unsqueeze(1), float("inf"))
        D[:, :, :per].diagonal(dim1=1, dim2=2).fill_(float("inf"))
        w, j = torch.topk(D, min(Kc, P * per - 1), dim=2, largest=False)
        t = torch.gather(pl.unsqueeze(1).expand(-1, per, -1), 2, j).reshape(-1, j.shape[2])
        rows = real[places[c:c + step]].reshape(-1)
        own.append(ids[places[c:c + step].reshape(-1)[rows]])
        tgt.append(ids[t[rows]])
        dst.append(w.reshape(-1, j.shape[2])[rows].clamp_min(0.0))
    own, tgt, dst = torch.cat(own), torch.cat(tgt), torch.cat(dst)
    tgt = torch.where(torch.isfinite(dst), tgt, -1)
    kept = _prune(X, dst, tgt, R)
    nbrs = _union(n, R, own.unsqueeze(1).expand_as(tgt)[kept], tgt[kept], dst[kept])
    # long links: half the slots of a random sample (ids are in random order) lead to its own graph
    s = min(n // 2, 4096)
    far = _layer(X[:s], R // 2)
    nbrs[:s] = torch.cat([far, nbrs[:s, :R - R // 2]], 1)
    entry = int(((X[:s] - X.mean(0)) ** 2).sum(1).argmin())
    return X, nbrs.contiguous(), entry, more


def _hierarchy(X, gen):
    """Upper layers of n/8, n/64, ... nodes: nested random subsets down to 16 nodes."""
    layers, ids = [], torch.arange(len(X), device="cuda")
    while len(ids) >= 128:
        pick = torch.randperm(len(ids), device="cuda", generator=gen)[:len(ids) // 8].sort().values
        ids = ids[pick]
        layer = dict(ids=ids, nbrs=_layer(X[ids], min(16, len(ids) - 1)))
        if layers:
            layer["down"] = pick
        layers.append({k: v.cpu().numpy() for k, v in layer.items()})
    return peos.Hierarchy(layers[::-1], 0)


# ------------------------------------------------------------------------------ cases
def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind, recipe, n = case["kind"], case["recipe"], case["n"]
    if kind in ("knn", "knn_tensor"):
        base, more = _points(recipe, n, gen)
        X = base.view(-1, base.shape[2])
        X = X[torch.randperm(len(X), device="cuda", generator=gen)[:n]].contiguous()
        return dict(case=case, X=X, Q=more(case["nq"]))
    X, nbrs, entry, more = _graph(recipe, n, gen)
    graph = peos.Graph(nbrs, entry)
    st = dict(case=case, X=X, graph=graph)
    if kind == "build":
        return st
    nq = case["nq"]
    st["codes"] = peos.build_codes(graph, X, RECIPES[recipe]["L"], M, PROJ_SEED) if case["routing"] else None
    storage = case.get("storage", "f32")
    st["base"] = X if storage == "f32" else peos.quantize(X, storage)
    st["opts"] = dict(eps=0.2, routing=case["routing"], eta_mode=1, beam=case.get("beam", 1))
    if case.get("rerank"):
        st["rerank"] = X
    Q = more(nq)
    st["Q"] = Q.cpu().numpy() if kind == "host" else Q
    if kind == "hier":
        st["layers"] = _hierarchy(X, gen)
    if kind == "batch":
        ef = torch.randint(min(32, case["ef"]), case["ef"] + 1, (nq,), device="cuda", generator=gen)
        ks = torch.tensor([1, min(10, case["k"]), case["k"]], device="cuda")
        k = ks[torch.randint(3, (nq,), device="cuda", generator=gen)]
        st["ef_q"], st["k_q"] = torch.maximum(ef, k).int(), k.int()
        size = peos.batch_workspace_size(graph, st["codes"], st["base"], nq, case["k"], case["ef"],
                                         rerank=st.get("rerank"), **st["opts"])
        st["workspace"] = torch.empty(size, dtype=torch.uint8, device="cuda")
        st["out"] = (torch.empty(nq, case["k"], dtype=torch.int32, device="cuda"),
                     torch.empty(nq, case["k"], dtype=torch.float32, device="cuda"), None)
    return st


class _Device:
    """A device array owned by an index, for torch to look at without a copy: the tensor
    keeps this object, and with it the index."""

    def __init__(self, codes, ptr, shape, typestr):
        self.codes = codes
        self.__cuda_array_interface__ = dict(data=(int(ptr), False), shape=tuple(shape), typestr=typestr, version=3)


def _index_arrays(codes):
    i = codes.info()
    n, R, sb = i["n"], i["R"], i["scalar_bits"]
    rec = torch.as_tensor(_Device(codes, i["records"], (n, i["record_stride"]), "|u1"), device="cuda")
    out = dict(records=rec,
               tables=torch.as_tensor(_Device(codes, i["node_proj"], (n, i["node_proj_stride"]), "<f4"), device="cuda"),
               norms=torch.as_tensor(_Device(codes, i["norms"], (n,), "<f4"), device="cuda"))
    if sb == 32:  # (||e||, w_reg, sqrt(L) w_res, node term) of each edge
        f = rec.view(torch.float32)
        out.update(e_norm=f[:, 0:4 * R:4], w_reg=f[:, 1:4 * R:4], c_res=f[:, 2:4 * R:4])
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "knn":
        return peos.knn_bruteforce(state["X"], state["Q"], case["k"])
    if kind == "knn_tensor":
        return peos.knn_tensor(state["X"], state["Q"], case["k"])
    graph = state["graph"]
    if kind == "build":
        return _index_arrays(peos.build_codes(graph, state["X"], RECIPES[case["recipe"]]["L"], M, PROJ_SEED,
                                              scalar_bits=case.get("scalar_bits", 32)))
    codes, base, Q, opts = state["codes"], state["base"], state["Q"], state["opts"]
    if kind == "host":
        return peos.search_host(graph, codes, base, Q, case["k"], case["ef"], **opts)[:2]
    if kind == "hier":
        entries = peos.hier_entry(state["layers"], base, Q)
        return (entries, *peos.search(graph, codes, base, Q, case["k"], case["ef"], entries=entries, **opts)[:2])
    if kind == "batch":
        return peos.search_batch(graph, codes, base, Q, case["k"], case["ef"], k_per_query=state["k_q"],
                                 ef_per_query=state["ef_q"], workspace=state["workspace"], out=state["out"],
                                 rerank=state.get("rerank"), **opts)[:2]
    return peos.search(graph, codes, base, Q, case["k"], case["ef"], rerank=state.get("rerank"), **opts)[:2]


def work(case):
    """Bytes and operations of one pass.  A search reads, per expansion, the node's edge
    record (28 bytes an edge; the ids alone without the test) and a row per exact distance;
    a list of ef takes about ef + 8 expansions, with about 10 exact distances each under the
    test and 14 without (a batch's lists are half its largest on average)."""
    r = RECIPES[case["recipe"]]
    n, d, R, L = case["n"], r["d"], r["R"], r["L"]
    kind = case["kind"]
    if kind in ("knn", "knn_tensor"):
        nq = case["nq"]
        return dict(bytes=4 * d * (n + nq) + 8 * nq * case["k"], flops=2 * n * nq * d)
    if kind == "build":
        degree = 14  # edges of a node, of its R slots
        sb = case.get("scalar_bits", 32)
        record = (28 if sb == 32 else 24 if sb == 16 else 20) * R + (0 if sb == 32 else 16)
        return dict(bytes=n * (4 * d + 4 * R + record + 4 * (L + 1) * M + 4), flops=n * (degree + 1) * 4 * d * M)
    nq, plain = case["nq"], case["routing"] == 0
    ef = case["ef"] / 2 if kind == "batch" else case["ef"]
    width = {"bf16": 2, "e4m3": 1}.get(case.get("storage"), 4)
    expansions = ef + 8
    dists = expansions * (14 if plain else 10)
    per = expansions * (4 if plain else 28) * R + dists * d * width + 4 * d + 8 * case["k"]
    per += ef * 4 * d if case.get("rerank") else 0
    return dict(bytes=nq * per, flops=nq * (3 * d * dists + (0 if plain else expansions * R * (L + 12))))


# ------------------------------------------------------------------- values in 64 bits
def exact(case, seed):
    """The brute force's distances, and the edge scalars and norms of an index.  What a graph
    search visits is decided step by step, so its results have no value of their own."""
    kind = case["kind"]
    if kind in ("knn", "knn_tensor"):
        st = prepare(case, seed)
        X, Q, k = st["X"], st["Q"], case["k"]
        sq = (X * X).sum(1)
        out = torch.empty(len(Q), k, dtype=torch.float64, device="cuda")
        for s in range(0, len(Q), 500):
            q = Q[s:s + 500]
            c = torch.topk(sq - 2.0 * (q @ X.T), min(len(X), k + 64), largest=False).indices
            d = torch.stack([((X[i].double() - v.double()) ** 2).sum(1) for i, v in zip(c, q)])
            out[s:s + 500] = d.sort(1).values[:, :k]
        return None, out
    if kind == "build":
        st = prepare(case, seed)
        X, nbrs, L = st["X"], st["graph"].nbrs, RECIPES[case["recipe"]]["L"]
        n, R = nbrs.shape
        norms = torch.cat([(x.double() ** 2).sum(1) for x in X.split(65536)])
        out = dict(records=None, tables=None, norms=norms)
        if case.get("scalar_bits", 32) == 32:
            parts = []
            for s in range(0, n, max(1, (1 << 26) // (R * X.shape[1]))):
                ids = nbrs[s:s + max(1, (1 << 26) // (R * X.shape[1]))].long()
                e = X[ids.clamp_min(0)].double() - X[s:s + len(ids)].double().unsqueeze(1)
                b = e.view(*e.shape[:2], L, -1).norm(dim=3)
                norm = b.square().sum(2).sqrt()
                w = torch.where(norm > 0, b.sum(2) / (math.sqrt(L) * norm), 1.0).clamp_max(1.0)
                c = math.sqrt(L) * (1.0 - w * w).clamp_min(0.0).sqrt()
                parts.append(torch.stack([norm, w, c]) * (ids >= 0))
            out["e_norm"], out["w_reg"], out["c_res"] = torch.cat(parts, 1)
        return out
    return None
