"""What users of the library have it do, as cases that can be timed.

Every case is one batch (a build, a kNN call or a range call) through the
public Python entry points, at the sizes of this repository's workloads or
scaled versions of them.  ``prepare`` makes what a program holds before the
call (objects and queries on the GPU, the built index), ``run`` makes the call
and takes its whole answer, ``exact`` gives the answer's distances by brute
force in FP64 with plain torch.

Families
  gauss    vectors from 64 isotropic Gaussians (embeddings with clusters)
  uniform  vectors uniform in [0, 1] (L1: colour-histogram-like features that
           no bound prunes)
  wordvec  anisotropic topic vectors under the angle (word embeddings)
  points   2 to 16-dimensional clustered points (locations, small features)
  words    random lower-case words and their misspellings (edit distance)
  dna      ACGT reads of length 108 around common seeds (edit distance)
  build    index construction
"""
import math
import statistics

import numpy as np
import torch

import paper_2404_00966_gb300 as gts


def listed():
    return [
        # an interactive lookup: one query against a mid-sized embedding set, all defaults
        dict(name="one_query_knn", family="gauss", op="knn", n=100_000, dim=128, nq=1, k=10, precision="fp32",
             fanout=20, n_pivots=0, metric="l2"),
        # spell checking: a small batch of words against a dictionary, range 2 (launch-bound)
        dict(name="words_range", family="words", op="range", n=10_000, nq=256, radius=2.0, precision="fp32",
             fanout=8, n_pivots=5, metric="edit"),
        # spelling suggestions: the five nearest dictionary words of a page of text
        dict(name="words_knn", family="words", op="knn", n=50_000, nq=999, k=5, precision="bf16", fanout=20,
             n_pivots=0, metric="edit"),
        # a large offline embedding join on the tensor-core path (the headline workload)
        dict(name="gauss_knn_bf16", family="gauss", op="knn", n=1_000_000, dim=128, nq=10_000, k=10,
             precision="bf16", fanout=20, n_pivots=0, metric="l2"),
        # the same data by a user who keeps the default precision
        dict(name="gauss_knn_fp32", family="gauss", op="knn", n=1_000_000, dim=128, nq=2_000, k=10,
             precision="fp32", fanout=20, n_pivots=0, metric="l2"),
        # near-duplicate search: all objects within a radius, ragged sizes
        dict(name="gauss_range_bf16", family="gauss", op="range", n=300_007, dim=100, nq=3_001, per_query=50,
             precision="bf16", fanout=20, n_pivots=0, metric="l2"),
        # angular nearest neighbours of word embeddings
        dict(name="wordvec_knn", family="wordvec", op="knn", n=200_000, dim=300, nq=10_000, k=10,
             precision="bf16", fanout=20, n_pivots=3, metric="cos"),
        # one serving batch of image-feature lookups under L1, k up to 100
        dict(name="l1_knn_batch", family="uniform", op="knn", n=2_000_000, dim=256, nq=128, k=100, mixed_k=True,
             precision="bf16", fanout=20, n_pivots=0, metric="l1"),
        # map service: all places near each of 10,000 positions, 10 M places
        dict(name="points_range", family="points", op="range", n=10_000_000, dim=2, nq=10_000, per_query=1000,
             precision="bf16", fanout=20, n_pivots=0, metric="l2"),
        # nearest stations / particles: small-dimensional kNN with the defaults
        dict(name="points_knn", family="points", op="knn", n=1_000_000, dim=3, nq=5_000, k=8, precision="fp32",
             fanout=20, n_pivots=0, metric="l2"),
        # read clustering: all reads within 8 edits of each of 20,000 reads, 1 M reads
        dict(name="dna_range", family="dna", op="range", n=1_000_000, nq=20_000, radius=8.0, precision="bf16",
             fanout=20, n_pivots=0, metric="edit"),
        # indexing a new collection that is already on the GPU
        dict(name="build_1M", family="build", op="build", n=1_000_000, dim=128, fanout=20, n_pivots=0, metric="l2"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    fam = rng.choice(["gauss", "gauss", "gauss", "uniform", "wordvec", "points", "points", "words", "dna", "build"])
    prec = rng.choice(["fp32", "bf16"])
    if fam == "build":
        dim = rng.choice([2, 3, 24, 100, 128])
        return dict(family="build", op="build", n=_log(rng, 20_000, 1_000_000), dim=dim, fanout=rng.choice([8, 20, 32]),
                    n_pivots=0, metric=rng.choice(["l2", "l1"]))
    if fam in ("words", "dna"):
        op = rng.choice(["range", "knn"])
        if fam == "words":
            c = dict(family=fam, op=op, n=_log(rng, 5_000, 200_000), nq=_log(rng, 1, 2_000), precision=prec,
                     fanout=rng.choice([8, 20]), n_pivots=0, metric="edit")
            c.update(radius=float(rng.choice([1, 2, 3])) if op == "range" else 0.0, k=rng.randint(1, 20))
        else:
            n = _log(rng, 20_000, 500_000)
            c = dict(family=fam, op=op, n=n, nq=_log(rng, 8, 5_000) if op == "range" else _log(rng, 8, 500),
                     precision=prec, fanout=20, n_pivots=0, metric="edit")
            c.update(radius=float(rng.randint(3, 9)) if op == "range" else 0.0, k=rng.randint(1, 16))
        return c
    if fam == "points":
        op = rng.choice(["range", "knn"])
        return dict(family=fam, op=op, n=_log(rng, 20_000, 5_000_000), dim=rng.choice([2, 2, 3, 5, 8]),
                    nq=_log(rng, 1, 5_000), k=_log(rng, 1, 64), per_query=_log(rng, 10, 1000), precision=prec,
                    fanout=rng.choice([8, 20, 20]), n_pivots=0, metric=rng.choice(["l2", "l2", "l1"]))
    if fam == "uniform":
        dim = rng.choice([64, 100, 192, 256])
        nq = _log(rng, 4, 192)
        n = min(_log(rng, 20_000, 1_000_000), int(2.5e10 / (dim * nq)))
        return dict(family=fam, op=rng.choice(["range", "knn"]), n=n, dim=dim, nq=nq, k=rng.randint(1, 100),
                    per_query=100, mixed_k=True, precision=prec, fanout=20, n_pivots=0, metric="l1")
    if fam == "wordvec":
        nq = _log(rng, 64, 10_000)
        return dict(family=fam, op=rng.choice(["range", "knn"]), n=_log(rng, 20_000, 200_000),
                    dim=rng.choice([96, 200, 300]), nq=nq, k=_log(rng, 1, 50), per_query=20, precision="bf16",
                    fanout=20, n_pivots=rng.choice([0, 3]), metric="cos")
    dim = rng.choice([17, 32, 48, 96, 100, 128, 128, 200, 256])
    nq = _log(rng, 1, 10_000)
    n = _log(rng, 10_000, 1_000_000)
    n = max(10_000, min(n, int((6e11 if prec == "bf16" else 1.2e11) / (dim * nq))))
    return dict(family="gauss", op=rng.choice(["range", "knn", "knn"]), n=n, dim=dim, nq=nq, k=_log(rng, 1, 100),
                per_query=_log(rng, 10, 300), precision=prec, fanout=rng.choice([8, 20, 20]), n_pivots=0,
                metric=rng.choice(["l2", "l2", "l2", "l1"]))


# ---------------------------------------------------------------- inputs

_CLUSTERS = {"gauss": 64, "wordvec": 500}


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda")


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _randint(g, lo, hi, *shape):
    return torch.randint(lo, hi, shape, generator=g, device="cuda")


def _vectors(case, seed):
    """Objects and queries, float32 on the GPU."""
    g = _gen(seed)
    n, dim, nq, fam = case["n"], case["dim"], case.get("nq", 0), case["family"]
    if fam == "uniform":
        return _rand(g, n, dim), _rand(g, nq, dim)
    if fam == "wordvec":
        scale = (torch.arange(dim, device="cuda", dtype=torch.float32) + 1.0) ** -0.3
        mean = 0.5 * _randn(g, dim) * scale
        centers = _randn(g, _CLUSTERS[fam], dim) * scale

        def some(m):
            return mean + centers[_randint(g, 0, _CLUSTERS[fam], m)] + 0.6 * _randn(g, m, dim) * scale
        return some(n), some(nq)
    if fam == "points" or (fam == "build" and dim <= 16):
        # 1,000 clusters with Zipf(1.1) weights
        centers = _rand(g, 1000, dim)
        w = torch.arange(1, 1001, device="cuda", dtype=torch.float64) ** -1.1
        cdf = torch.cumsum(w / w.sum(), 0)

        def some(m):
            lab = torch.searchsorted(cdf, torch.rand(m, generator=g, device="cuda", dtype=torch.float64))
            return centers[lab.clamp_(max=999)] + 0.01 * _randn(g, m, dim)
        return some(n), some(nq)
    centers = 2.0 * _rand(g, 64, dim) - 1.0

    def some(m):
        return _randn(g, m, dim).mul_(0.1).add_(centers[_randint(g, 0, 64, m)])
    return some(n), some(nq)


def _edit_rows(g, mat, length, edits, alphabet):
    """Random unit edits on padded strings: mat uint8 [n, L], length int64 [n], edits int64 [n]."""
    n, L = mat.shape
    cols = torch.arange(L, device="cuda")[None, :]
    for e in range(int(edits.max())):
        op = _randint(g, 0, 3, n)                                   # 0 substitute, 1 insert, 2 delete
        op = torch.where((op == 2) & (length <= 1), torch.zeros_like(op), op)
        op = torch.where(edits > e, op, torch.full_like(op, 3))
        span = length + (op == 1).long()
        at = (_rand(g, n).double() * span).long().clamp_(max=L - 1)[:, None]
        letter = alphabet[_randint(g, 0, alphabet.numel(), n)][:, None].expand(n, L)
        ins, dele = (op == 1)[:, None], (op == 2)[:, None]
        src = cols - (ins & (cols > at)).long() + (dele & (cols >= at)).long()
        mat = torch.gather(mat, 1, src.clamp_(0, L - 1))
        put = (cols == at) & (op <= 1)[:, None]
        mat = torch.where(put, letter, mat)
        length = length + (op == 1).long() - (op == 2).long()
    return mat, length


def _pack(mat, length):
    """Padded strings to (bytes, offsets)."""
    keep = torch.arange(mat.shape[1], device="cuda")[None, :] < length[:, None]
    offsets = torch.zeros(length.numel() + 1, dtype=torch.int64, device="cuda")
    offsets[1:] = torch.cumsum(length, 0)
    return mat[keep].contiguous(), offsets


def _string_rows(case, seed):
    """Objects and queries as padded rows with lengths."""
    g = _gen(seed)
    n, nq = case["n"], case["nq"]
    if case["family"] == "words":
        alphabet = torch.arange(97, 123, device="cuda", dtype=torch.uint8)
        length = _randint(g, 4, 17, n)
        mat = alphabet[_randint(g, 0, 26, n, 20)]
        pick = _randint(g, 0, n, nq)
        q, ql = _edit_rows(g, mat[pick], length[pick], _randint(g, 0, 4, nq), alphabet)
        return mat, length, q, ql
    alphabet = torch.tensor([65, 67, 71, 84], device="cuda", dtype=torch.uint8)
    seeds = max(1, n // 100)
    base = alphabet[_randint(g, 0, 4, seeds, 116)]
    lab = torch.arange(n, device="cuda") % seeds
    full = torch.full((n,), 108, dtype=torch.int64, device="cuda")
    mat, length = _edit_rows(g, base[lab], full, _randint(g, 1, 7, n), alphabet)
    pick = _randint(g, 0, seeds, nq)
    q, ql = _edit_rows(g, base[pick], full[:1].expand(nq), _randint(g, 1, 7, nq), alphabet)
    return mat, length, q, ql


def _k(case, seed):
    """int32[nq] on the GPU; mixed_k: 1 .. k spread evenly over the batch, in random order."""
    if case.get("mixed_k"):
        nq = case["nq"]
        order = torch.randperm(nq, generator=_gen(seed + 7919), device="cuda")
        return (1 + order * case["k"] // nq).to(torch.int32)
    return torch.full((case["nq"],), case["k"], dtype=torch.int32, device="cuda")


def _radius(case, X, Q):
    """A radius with about `per_query` answers per query (float)."""
    if "radius" in case and case["metric"] == "edit":
        return float(case["radius"])
    n, dim, want = case["n"], case["dim"], case["per_query"]
    p = min(0.5, want / n)
    if case["family"] == "uniform":       # a sum of dim coordinates |x - y|, mean 1/3, variance 1/18
        return dim / 3.0 + statistics.NormalDist().inv_cdf(p) * math.sqrt(dim / 18.0)
    if case["family"] == "gauss":         # within the query's cluster: sigma^2 sums of dim terms
        z = statistics.NormalDist().inv_cdf(min(0.5, p * _CLUSTERS["gauss"]))
        if case["metric"] == "l1":        # |x - y| of N(0, 2 sigma^2): mean 2 sigma / sqrt(pi)
            s = 0.1 * math.sqrt(2.0)
            return s * (dim * math.sqrt(2.0 / math.pi) + z * math.sqrt(dim * (1.0 - 2.0 / math.pi)))
        return math.sqrt(0.02 * dim * max(0.05, 1.0 - 2.0 / (9 * dim) + z * math.sqrt(2.0 / (9 * dim))) ** 3)
    # points, wordvec: the quantile of a sample's distances
    xs, qs = X[:400_000].double(), Q[:64].double()
    if case["metric"] == "cos":
        d = torch.acos((torch.nn.functional.normalize(qs) @ torch.nn.functional.normalize(xs).T).clamp(-1, 1))
    else:
        d = torch.cdist(qs, xs, p=1.0 if case["metric"] == "l1" else 2.0,
                        compute_mode="donot_use_mm_for_euclid_dist")
    kth = max(1, int(round(p * d.numel())))
    return float(torch.kthvalue(d.reshape(-1), kth).values)


def _capacity(case):
    """Answers a range program keeps room for (its result buffers are made once)."""
    nq, n = case["nq"], case["n"]
    if case["family"] == "words":
        per = max(64, n // 50)
    elif case["family"] == "dna":
        per = 128
    else:
        per = min(n, 6 * case["per_query"] + 64)
    return nq * per + 4096


def prepare(case, seed):
    op = case["op"]
    if case["metric"] == "edit":
        mat, length, q, ql = _string_rows(case, seed)
        objects, queries = _pack(mat, length), _pack(q, ql)
        X = Q = None
    else:
        X, Q = _vectors(case, seed)
        objects, queries = X, Q
    if op == "build":
        return dict(op=op, objects=objects, case=case)
    index = gts.Index.build(objects, case["metric"], n_pivots=case["n_pivots"], fanout=case["fanout"], root_pivot=0)
    if op == "knn":
        per = _k(case, seed)
    else:
        per = torch.full((case["nq"],), _radius(case, X, Q), dtype=torch.float32, device="cuda")
    state = dict(op=op, index=index, queries=queries, per=per, precision=case["precision"], case=case)
    total = int(per.sum()) if op == "knn" else _capacity(case)
    if case["nq"] < 2000:     # small batches: the answers come to the host (the default)
        if op == "range":
            state.update(ids=np.full(total, -1, np.int64), dist=np.full(total, -1.0, np.float32))
    else:                     # large ones stay on the GPU
        state.update(offsets=torch.zeros(case["nq"] + 1, dtype=torch.int64, device="cuda"),
                     ids=torch.full((total,), -1, dtype=torch.int64, device="cuda"),
                     dist=torch.full((total,), -1.0, dtype=torch.float32, device="cuda"))
    return state


# ---------------------------------------------------------------- the call

def run(state):
    if state["op"] == "build":
        c = state["case"]
        index = gts.Index.build(state["objects"], c["metric"], n_pivots=c["n_pivots"], fanout=c["fanout"],
                                root_pivot=0)
        ids, table = index.table()
        index.close()
        return [ids, table]
    call = state["index"].knn if state["op"] == "knn" else state["index"].range
    if "offsets" not in state:
        r = call(state["queries"], state["per"], precision=state["precision"])
        if state["op"] == "knn":
            return [r.offsets, r.ids, r.dist]
        m = r.ids.shape[0]
        state["ids"][:m] = r.ids
        state["dist"][:m] = r.dist
        return [r.offsets, state["ids"], state["dist"]]
    r = call(state["queries"], state["per"], precision=state["precision"], result_on_device=True)
    if r.stats["results"] > state["ids"].numel():
        raise ValueError("more answers than the program keeps room for")
    r.copy_to(state["offsets"], state["ids"], state["dist"])
    r.free()
    return [state["offsets"], state["ids"], state["dist"]]


# ---------------------------------------------------------------- what a pass cannot do without

def work(case):
    """Each object and query read once, each answer written once; arithmetic of
    the pairs that no metric bound of these data excludes (a query against its
    own cluster; against everything where distances concentrate)."""
    n, nq = case["n"], case.get("nq", 0)
    row = 108 if case["family"] == "dna" else 10 if case["family"] == "words" else 4 * case["dim"]
    if case["op"] == "build":
        h = max(1, math.ceil(math.log(n + 1) / math.log(case["fanout"])) - 1)
        return {"bytes": n * (row + row + 4 * h + 8), "flops": 3 * case["dim"] * n * h}
    if case["op"] == "knn":
        answers = nq * min(n, case["k"])
    else:
        answers = nq * min(n, case.get("per_query", 100 if case["family"] == "dna" else 5))
    pairs = answers
    if case["family"] in _CLUSTERS:
        pairs = max(answers, nq * (n // _CLUSTERS[case["family"]]))
    elif case["family"] == "uniform":
        pairs = nq * n
    elif case["family"] == "dna":
        pairs = nq * 100
    if case["metric"] == "edit":        # bit-parallel: about 10 operations per 32 cells
        flops = pairs * row * 10 * ((row + 31) // 32)
    else:
        flops = pairs * 2 * case["dim"]
    return {"bytes": n * row + nq * row + answers * 12 + nq * 8, "flops": flops}


# ---------------------------------------------------------------- exact distances, brute force in FP64

def _pair_dist(metric, q, x):
    """FP64 distances of paired rows [m, dim]."""
    if metric == "l1":
        return (q - x).abs().sum(1)
    if metric == "cos":
        return torch.acos(((q * x).sum(1) / (q.norm(dim=1) * x.norm(dim=1))).clamp(-1, 1))
    return (q - x).square().sum(1).sqrt()


def _chunks(case, X, Q):
    """Per chunk of queries: (first query, [m, n] FP64 values ordered like the distances, their scale's meaning)."""
    n, nq, dim, metric = case["n"], case["nq"], case["dim"], case["metric"]
    step = max(1, min(nq, int(4e8 / n)))
    Xd = torch.nn.functional.normalize(X) if metric == "cos" else X
    Qd = torch.nn.functional.normalize(Q) if metric == "cos" else Q
    x2 = Xd.square().sum(1)
    for s in range(0, nq, step):
        q = Qd[s:s + step]
        if metric == "l1" or dim <= 16:
            v = torch.zeros(q.shape[0], n, dtype=torch.float64, device="cuda")
            if metric == "l1" and dim > 16:
                for i in range(q.shape[0]):
                    for a in range(0, n, 1 << 20):
                        v[i, a:a + (1 << 20)] = (Xd[a:a + (1 << 20)] - q[i]).abs().sum(1)
            else:
                for j in range(dim):
                    t = q[:, j, None] - Xd[None, :, j]
                    v += t.abs() if metric == "l1" else t * t
            yield s, (v if metric == "l1" else v.sqrt_())
        else:
            v = torch.addmm(x2[None, :].expand(q.shape[0], n), q, Xd.T, alpha=-2.0)
            v += q.square().sum(1)[:, None]
            yield s, v.clamp_(min=0.0).sqrt_()


def _laid_out(case, parts):
    """The distances as run() lays them out (range: in the program's buffer)."""
    d = torch.cat(parts)
    if case["op"] == "range":
        buf = torch.full((_capacity(case),), -1.0, dtype=torch.float64, device="cuda")
        buf[:d.numel()] = d
        d = buf
    return [None, None, d]


def _exact_vec(case, seed):
    X, Q = _vectors(case, seed)
    radius = None if case["op"] == "knn" else torch.tensor(_radius(case, X, Q), dtype=torch.float32).double().item()
    X, Q = X.double(), Q.double()
    metric = case["metric"]
    out = []
    if case["op"] == "knn":
        k = _k(case, seed).long()
        top = min(case["n"], int(k.max()) + 8)
        for s, v in _chunks(case, X, Q):
            m = v.shape[0]
            near = torch.topk(v, top, dim=1, largest=False).indices
            d = _pair_dist(metric, Q[s:s + m].repeat_interleave(top, 0), X[near.reshape(-1)]).reshape(m, top)
            d = d.sort(dim=1).values
            keep = torch.arange(top, device="cuda")[None, :] < k[s:s + m, None]
            out.append(d[keep])
    else:
        lim = 2.0 * math.sin(min(radius, math.pi) / 2.0) if metric == "cos" else radius
        for s, v in _chunks(case, X, Q):
            hit = torch.nonzero(v <= lim)
            for a in range(0, hit.shape[0], 1 << 20):
                h = hit[a:a + (1 << 20)]
                out.append(_pair_dist(metric, Q[s + h[:, 0]], X[h[:, 1]]))
    return _laid_out(case, out)


def _exact_words(case, seed):
    """Every pair's Levenshtein distance, a row of the DP at a time for all pairs of a query."""
    mat, length, q, ql = _string_rows(case, seed)
    n, cols = mat.shape
    out = []
    for i in range(case["nq"]):
        row = torch.arange(cols + 1, device="cuda", dtype=torch.int32)[None, :].repeat(n, 1)
        ar = torch.arange(cols + 1, device="cuda", dtype=torch.int32)[None, :]
        for a in range(int(ql[i])):
            sub = row[:, :-1] + (mat != q[i, a]).int()
            best = torch.minimum(sub, row[:, 1:] + 1)
            best = torch.cat([row[:, :1] + 1, best], 1)
            row = torch.cummin(best - ar, 1).values + ar
        d = row.gather(1, length[:, None])[:, 0].double()
        if case["op"] == "knn":
            out.append(d.sort().values[:min(n, case["k"])])
        else:
            out.append(d[d <= math.floor(case["radius"])])
    return _laid_out(case, out)


def exact(case, seed):
    if case["op"] == "build":
        return None       # the tree's layout follows the build's own FP32 distances
    if case["metric"] == "edit":
        small = case["family"] == "words" and case["n"] * case["nq"] <= 6e7
        return _exact_words(case, seed) if small else None
    return _exact_vec(case, seed)
