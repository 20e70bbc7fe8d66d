"""What a program that uses this library has it do, as cases that can be timed and compared.

Sizes are those of the library's named workloads (tiny, medium, precision, batching, tail, beam, the
ordering MLP's training step) and of its ragged and constrained tests.  The graphs are R-MAT or Zipf typed
knowledge graphs like those of the synthetic workloads, made on the GPU from the seed.

Families:
  one     one query, synchronous, host arrays in and out (a lookup service's single request)
  batch   a batch of three-hop queries on device arrays (the library's main path)
  noalloc one query through the entry point for callers that cannot allocate
  tail    tail prediction: heads against every vertex of a type, or against every vertex
  beam    H-hop beam search
  mlp     one training step of the ordering MLP: features, forward, backward, Adam, bf16 weights
  edges   edge weights of the graph's edges or of given triples
  load    graph load followed by the first batch (start-up of a service, a one-off analysis)
"""

import math

import numpy as np
import torch

import paper_2406_07727_gb300 as mhr

DEV = "cuda"


def listed():
    return [
        # smallest call: one hub-to-hub question on a small graph; latency and launches
        _graph("one_tiny", "one", kind="zipf", n=10_000, E=100_000, R=8, types=4, d=64, nq=1, K=10, queries="hub"),
        # a service's ordinary batch with the default options
        _graph("batch_medium_plain", "batch", n=1_000_000, E=20_000_000, R=16, types=6, d=128, nq=64, K=100),
        # DistMult on wide rows, ordered by bound and pruned: an interactive service's batch
        _graph("batch_precision_bound", "batch", n=1_000_000, E=20_000_000, R=16, types=6, d=256, nq=256, K=100,
               score="distmult", order=1, prune=1),
        # odd sizes: a row length no vector load divides, a ragged batch, one relation set per hop and typed
        # intermediate vertices (the constrained query shape)
        _graph("batch_ragged_constrained", "batch", n=77_777, E=1_234_567, R=11, types=5, d=50, nq=37, K=33,
               constrained=1),
        # the largest batch one GPU is asked for: 4,096 queries on 10M vertices, bf16 rows, ordered and pruned
        _graph("batch_large_bf16", "batch", n=10_000_000, E=200_000_000, R=32, types=6, d=128, dtype="bf16", nq=4096,
               K=50, order=1, prune=1, queries="logdeg"),
        # one query in a section that cannot allocate
        _graph("noalloc_small", "noalloc", n=100_000, E=1_000_000, R=8, types=4, d=64, nq=1, K=20),
        # tail prediction, many heads against one type (every university of one person, batched over persons)
        _graph("tail_typed", "tail", n=1_000_000, E=2_000_000, R=16, types=6, d=128, nq=64, K=50, cand=0),
        # tail prediction, one head against every vertex (every person for one award)
        _graph("tail_single", "tail", n=1_000_000, E=2_000_000, R=16, types=6, d=128, nq=1, K=50, cand=-1),
        # multi-hop beam search, a batch of queries
        _graph("beam_medium", "beam", n=1_000_000, E=20_000_000, R=16, types=6, d=128, nq=64, K=10, H=3),
        # one step of training the ordering network at the driver's batch size
        _graph("mlp_step", "mlp", n=1_000_000, E=2_000_000, R=16, types=6, d=256, rows=4096),
        # every edge of a graph scored (link scoring, export)
        _graph("edges_all", "edges", n=1_000_000, E=20_000_000, R=16, types=6, d=128, rows=0, precision=0),
        # start-up: graph load and the first batch of questions
        _graph("load_medium", "load", n=1_000_000, E=20_000_000, R=16, types=6, d=128, nq=16, K=50, order=1, prune=1),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    family = rng.choice(["one", "batch", "batch", "batch", "noalloc", "tail", "tail", "beam", "mlp", "edges", "load"])
    top = {"noalloc": 1_000_000, "mlp": 2_000_000, "tail": 4_000_000}.get(family, 20_000_000)
    E = log_int(50_000, top)
    n = max(2_000, E // rng.randint(8, 25)) if family != "tail" else log_int(10_000, 1_000_000)
    E = max(E, 2 * n)
    c = dict(n=n, E=E, R=rng.choice([1, 5, 8, 11, 16, 32]), types=rng.randint(1, 8),
             d=rng.choice([32, 50, 64, 100, 127, 128, 200, 256]), dtype=rng.choice(["f32", "bf16"]),
             score=rng.choice(["transe", "distmult"]), kind=rng.choice(["rmat", "rmat", "zipf"]))
    if family in ("batch", "load", "one"):
        c["order"] = c["prune"] = rng.choice([0, 1])
        c["K"] = log_int(1, 500 if family == "batch" else 100)
        c["nq"] = 1 if family == "one" else log_int(1, 512 if family == "batch" else 64)
        if family == "batch":
            c["constrained"] = rng.choice([0, 0, 0, 1])
            c["queries"] = rng.choice(["edge", "edge", "logdeg"])
    elif family == "noalloc":
        c["nq"], c["K"] = 1, log_int(1, 200)
    elif family == "tail":
        c["nq"], c["K"], c["cand"] = log_int(1, 256), log_int(1, 1000), rng.choice([-1, 0])
    elif family == "beam":
        c["H"] = rng.choice([2, 3, 4])
        c["K"] = rng.randint(2, {2: 64, 3: 20, 4: 8}[c["H"]])
        c["nq"] = log_int(1, 64)
    elif family == "mlp":
        c["rows"] = log_int(100, 131_072)
    else:
        c["rows"] = rng.choice([0, log_int(1_000, 5_000_000)])
        c["precision"] = rng.choice([0, 0, 2])
        if c["precision"] == 2 and not c["rows"]:
            c["rows"] = log_int(1_000, 5_000_000)
    return _graph(None, family, **c)


def _graph(name, family, **kw):
    """A case with every field filled in."""
    c = dict(family=family, kind="rmat", n=0, E=0, R=1, types=1, d=0, dtype="f32", score="transe", nq=1, K=1, H=0,
             order=0, prune=0, constrained=0, queries="edge", cand=-1, rows=0, precision=0)
    c.update(kw)
    return dict(name=name, **c) if name else c


# ----------------------------------------------------------------------------- inputs
def _edges(c, gen):
    """Sorted distinct (u, v, r) keys of c["E"] edges without self loops."""
    n, E, R = c["n"], c["E"], c["R"]
    scale = max(1, (n - 1).bit_length())
    keys = torch.empty(0, dtype=torch.int64, device=DEV)
    perm = torch.randperm(n, generator=gen, device=DEV)
    src = None
    if c["kind"] == "zipf":
        # out-degrees of a power law with exponent 2.1, scaled to the edge count
        f = (1.0 - torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)).pow(-1.0 / 1.1).clamp(max=n - 1)
        src = torch.cumsum(f / f.sum(), 0)
    while True:
        m = int((E - keys.numel()) * 1.7) + 4096
        if c["kind"] == "zipf":
            u = torch.searchsorted(src, torch.rand(m, generator=gen, device=DEV, dtype=torch.float64)).clamp(max=n - 1)
            v = torch.randint(0, n, (m,), generator=gen, device=DEV)
        else:
            # R-MAT quadrants (.57, .19, .19, .05); endpoints past n are dropped
            u = torch.zeros(m, dtype=torch.int64, device=DEV)
            v = torch.zeros(m, dtype=torch.int64, device=DEV)
            for _ in range(scale):
                q = torch.rand(m, generator=gen, device=DEV)
                u = u * 2 + (q >= 0.76)
                v = v * 2 + (((q >= 0.57) & (q < 0.76)) | (q >= 0.95))
                del q
        ok = (u < n) & (v < n) & (u != v)
        u, v = perm[u[ok]], perm[v[ok]]
        r = torch.randint(0, R, (u.numel(),), generator=gen, device=DEV)
        k = (u * n + v) * R + r
        del u, v, r, ok
        keys = torch.unique(torch.cat([keys, k]))
        del k
        if keys.numel() >= E:
            break
    if keys.numel() > E:  # an evenly spaced subset stays sorted
        keys = keys[torch.arange(E, device=DEV) * keys.numel() // E]
    return keys


def _arrays(c, seed):
    """The graph, embeddings and queries of a case, on the GPU."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    n, R, d = c["n"], c["R"], c["d"]
    keys = _edges(c, gen)
    A = {"rels": (keys % R).to(torch.int16)}
    uv = keys // R
    del keys
    A["cols"] = (uv % n).to(torch.int32)
    deg = torch.bincount(uv // n, minlength=n)
    del uv
    A["off"] = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(deg, 0)])
    A["vt"] = torch.randint(0, c["types"], (n,), generator=gen, device=DEV).to(torch.uint8)
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    std = d ** -0.25
    A["vemb"] = (torch.randn((n, d), generator=gen, device=DEV) * std).to(dt)
    A["remb"] = (torch.randn((R, d), generator=gen, device=DEV) * std).to(dt)
    E, nq = A["cols"].numel(), c["nq"]

    def source_of(e):
        return torch.searchsorted(A["off"], e, right=True) - 1

    if c["queries"] == "hub":
        S = deg.argmax().reshape(1)
        ind = torch.bincount(A["cols"], minlength=n)
        ind[S] = -1
        T = ind.argmax().reshape(1)
    else:
        T = A["cols"][torch.randint(0, E, (nq,), generator=gen, device=DEV)].to(torch.int64)
        if c["queries"] == "logdeg":
            # source degree log-uniform: a degree octave, then a vertex of it (the next lower octave that has one)
            octave = torch.floor(torch.log2(deg.clamp(min=1).to(torch.float64))).to(torch.int64)
            octave[deg == 0] = -1
            order = torch.argsort(octave, stable=True)
            cnt = torch.bincount(octave + 1, minlength=64)
            first = torch.cumsum(cnt, 0) - cnt
            have = torch.where(cnt > 0, torch.arange(cnt.numel(), device=DEV), torch.zeros_like(cnt)).cummax(0).values
            x = torch.rand(nq, generator=gen, device=DEV, dtype=torch.float64) * math.log2(1e5)
            b = have[torch.floor(x).to(torch.int64) + 1].clamp(min=1)
            pick = (torch.rand(nq, generator=gen, device=DEV, dtype=torch.float64) * cnt[b]).to(torch.int64)
            S = order[first[b] + torch.minimum(pick, cnt[b] - 1)]
        else:
            S = source_of(torch.randint(0, E, (nq,), generator=gen, device=DEV))
        T = torch.where(T == S, (T + 1) % n, T)
    A["S"], A["T"] = S.to(torch.int32), T.to(torch.int32)
    if c["family"] == "tail":
        A["S"] = torch.randint(0, n, (nq,), generator=gen, device=DEV).to(torch.int32)
        A["Rq"] = torch.randint(0, R, (nq,), generator=gen, device=DEV).to(torch.int16)
    if c["family"] == "mlp":
        m, g = c["rows"], gen
        A["va"] = torch.randint(0, n, (m,), generator=g, device=DEV).to(torch.int32)
        A["vb"] = torch.randint(0, n, (m,), generator=g, device=DEV).to(torch.int32)
        A["target"] = torch.randn(m, generator=g, device=DEV)
        A["params"] = torch.cat([torch.randn(256 * 256, generator=g, device=DEV) * math.sqrt(2 / 256),
                                 torch.randn(256, generator=g, device=DEV) * 0.05,
                                 torch.randn(256, generator=g, device=DEV) / 16,
                                 torch.randn(1, generator=g, device=DEV) * 0.05])
        # a step in the middle of training: moments of a hundred earlier steps
        A["m1"] = torch.randn(A["params"].numel(), generator=g, device=DEV) * 1e-3
        A["m2"] = torch.rand(A["params"].numel(), generator=g, device=DEV) * 1e-5 + 1e-7
    if c["family"] == "edges" and c["rows"]:
        A["src"] = torch.randint(0, n, (c["rows"],), generator=gen, device=DEV).to(torch.int32)
        A["dst"] = torch.randint(0, n, (c["rows"],), generator=gen, device=DEV).to(torch.int32)
        A["rq"] = torch.randint(0, R, (c["rows"],), generator=gen, device=DEV).to(torch.int16)
    return A


def _constraints(c):
    """About half of the relations per hop, a few types for u and v."""
    R, t = c["R"], c["types"]
    return {"rel1": list(range(0, R, 2)), "rel2": list(range(R // 3, R)), "rel3": list(range((R + 1) // 2)) or [0],
            "types_u": list(range(0, t, 2)), "types_v": list(range(t // 2, t))}


def _load(A, c):
    return mhr.mhr_graph_load(A["off"], A["cols"], A["rels"], A["vemb"], A["remb"], c["R"], vtypes=A["vt"],
                              n_vtypes=c["types"], score_fn=c["score"], emb_dtype=c["dtype"])


def prepare(case, seed):
    c, A = case, _arrays(case, seed)
    st = {"case": c, "S": A["S"], "T": A["T"], "rank": torch.arange(max(1, c["K"]), device=DEV)}
    st["opts"] = {"order": c["order"], "prune": c["prune"]} if c["order"] or c["prune"] else None
    if c["constrained"]:
        st["opts"] = dict(st["opts"] or {}, constraints=_constraints(c))
    if c["family"] == "load":
        st["A"] = A
        return st
    st["G"] = _load(A, c)
    if c["family"] in ("one", "noalloc"):
        st["s"], st["t"] = int(A["S"][0]), int(A["T"][0])
        st["out"] = torch.empty((1, c["K"] * mhr.PATH_DTYPE.itemsize), dtype=torch.uint8, device=DEV)
        st["n_out"] = torch.empty(1, dtype=torch.int32, device=DEV)
    elif c["family"] == "tail":
        st["Rq"] = A["Rq"]
    elif c["family"] == "mlp":
        rows = c["rows"]
        m = mhr.OrderingMLP(params=A["params"].cpu().numpy())
        m.m1.copy_(A["m1"])
        m.m2.copy_(A["m2"])
        m.step = 100
        st.update(model=m, va=A["va"], vb=A["vb"], target=A["target"],
                  y=torch.empty(rows, device=DEV), z1=torch.empty((rows, 256), device=DEV),
                  work=torch.empty((rows, 256), device=DEV), grads=torch.empty(m.params.numel(), device=DEV),
                  loss=torch.empty(1, device=DEV))
    elif c["family"] == "edges":
        n = c["rows"] or st["G"].E
        st["out"] = torch.empty(n, dtype=torch.float32 if c["precision"] == 0 else torch.float64, device=DEV)
        st["triples"] = (A["src"], A["rq"], A["dst"]) if c["rows"] else (None, None, None)
    torch.cuda.synchronize()
    return st


# ----------------------------------------------------------------------------- one pass
def _lists(st, out, n_out, K):
    """Score and id columns of the results, zero past each query's count."""
    nq = n_out.numel()
    words = out.view(torch.int64).view(nq, K, -1)
    live = st["rank"] < n_out[:, None]
    score = torch.where(live, out.view(torch.float64).view(nq, K, -1)[..., 0], 0.0)
    return {"score": score, "ids": torch.where(live[..., None], words[..., 1:], 0), "n": n_out}


def run(st):
    c = st["case"]
    f, K = c["family"], c["K"]
    if f == "one":
        p = mhr.mhr_topk_paths(st["G"], st["s"], st["t"], K, opts=st["opts"])
        return {k: p[k] for k in ("score", "u", "v", "r1", "r2", "r3")}
    if f == "batch":
        out, n = mhr.mhr_topk_paths_batched(st["G"], st["S"], st["T"], K, opts=st["opts"])
        return _lists(st, out, n, K)
    if f == "noalloc":
        mhr.mhr_topk_paths_noalloc(st["G"], st["s"], st["t"], K, st["out"], st["n_out"])
        return _lists(st, st["out"], st["n_out"], K)
    if f == "tail":
        out, n = mhr.mhr_tail_topk(st["G"], st["S"], st["Rq"], K, cand_type=c["cand"])
        return _lists(st, out, n, K)
    if f == "beam":
        out, n = mhr.mhr_beam_paths(st["G"], st["S"], st["T"], c["H"], K)
        return _lists(st, out, n, K)
    if f == "mlp":
        m = st["model"]
        X = mhr.mhr_mlp_features(st["G"], st["va"], st["vb"])
        mhr.mhr_mlp_forward(m, X, st["y"], st["z1"])
        mhr.mhr_mlp_backward(m, X, st["target"], st["y"], st["z1"], st["work"], st["grads"], st["loss"])
        m.step += 1
        mhr.mhr_mlp_adam(m.params, st["grads"], m.m1, m.m2, 1e-3, m.step)
        m.refresh()
        return {"X": X.view(torch.bfloat16), "y": st["y"], "z1": st["z1"], "grads": st["grads"], "loss": st["loss"],
                "params": m.params, "m1": m.m1, "m2": m.m2, "W1": m.W1b.view(torch.bfloat16)}
    if f == "edges":
        src, rel, dst = st["triples"]
        return {"w": mhr.mhr_edge_scores(st["G"], src, rel, dst, precision=c["precision"], out=st["out"])}
    G = _load(st["A"], c)
    out, n = mhr.mhr_topk_paths_batched(G, st["S"], st["T"], K, opts=st["opts"])
    r = _lists(st, out, n, K)
    mhr.mhr_graph_free(G)
    return r


# ----------------------------------------------------------------------------- work
def work(case):
    """Bytes and flops of one pass, each input read once.  What a search reads depends on the queries' degrees;
    a query is credited with the mean frontier and middle-edge counts of degree-biased endpoints (about 30 and
    900 mean degrees), never more than the graph holds."""
    c = case
    n, E, d, nq, K = c["n"], c["E"], c["d"], c["nq"], c["K"]
    es = 4 if c["dtype"] == "f32" else 2
    row, csr, deg = d * es, 6 * E + 8 * n, E / n
    f = c["family"]
    if f in ("one", "batch", "noalloc", "load"):
        front = nq * min(60.0 * deg, n)
        middle = nq * min(900.0 * deg * deg, E)
        b = min(6.0 * middle, csr) + min(front, n) * row + 24.0 * nq * K
        fl = 3.0 * d * (front + 0.05 * middle)
        if f == "load":
            b, fl = b + 2 * csr + 2.0 * n * row + E * 6, fl + 3.0 * d * E
        return {"bytes": b, "flops": fl}
    if f == "tail":
        cand = n if c["cand"] < 0 else n / c["types"]
        return {"bytes": cand * (row + 4.0) + 16.0 * nq * K, "flops": 2.0 * d * nq * cand}
    if f == "beam":
        held = nq * sum(K ** i for i in range(c["H"]))
        edges = held * min(60.0 * deg, n)
        return {"bytes": min(edges * 6.0, csr) + min(edges, n) * row + 64.0 * nq * K, "flops": 3.0 * d * edges}
    if f == "mlp":
        m, P = c["rows"], 256 * 256 + 513
        return {"bytes": m * (2.0 * 128 * es + 512 + 3 * 1024 + 16) + P * 30.0, "flops": 4.0 * m * 65536}
    m = c["rows"] or E
    touched = n if not c["rows"] else min(n, 2 * m)
    return {"bytes": m * (10.0 if c["rows"] else 6.0) + touched * row + m * (4.0 if c["precision"] == 0 else 8.0),
            "flops": 3.0 * d * m}


# ----------------------------------------------------------------------------- the same in 64 bits
class _Exact:
    """Plain torch definitions in float64 of what the library computes."""

    def __init__(self, c, A):
        self.c, self.A, self.n = c, A, c["n"]
        self.off, self.cols, self.rels = A["off"], A["cols"].to(torch.int64), A["rels"].to(torch.int64)

    def weight(self, h, r, t):
        """w(h, r, t) of index vectors: 1 - |e_h + w_r - e_t|_1, or the trilinear product."""
        out = torch.empty(h.numel(), dtype=torch.float64, device=DEV)
        step = max(1, (1 << 27) // self.c["d"])
        V, W = self.A["vemb"], self.A["remb"]
        for i in range(0, h.numel(), step):
            a, b, e = V[h[i:i + step]].double(), W[r[i:i + step]].double(), V[t[i:i + step]].double()
            out[i:i + step] = 1.0 - (a + b - e).abs().sum(1) if self.c["score"] == "transe" else (a * b * e).sum(1)
        return out

    def rows_of(self, x):
        """(position in x, edge index) of every out-edge of the vertices x."""
        lo, deg = self.off[x], self.off[x + 1] - self.off[x]
        own = torch.repeat_interleave(torch.arange(x.numel(), device=DEV), deg)
        first = torch.cumsum(deg, 0) - deg
        return own, lo[own] + torch.arange(own.numel(), device=DEV) - first[own]

    def reverse(self):
        self.rorder = torch.argsort(self.cols, stable=True)
        cnt = torch.bincount(self.cols, minlength=self.n)
        self.roff = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(cnt, 0)])
        self.rsrc = torch.searchsorted(self.off, self.rorder, right=True) - 1

    def paths(self, s, t, K, cons):
        """Scores of the K best simple three-hop paths, zero past the last one."""
        allow = {k: torch.zeros(max(256, self.c["R"]), dtype=torch.bool, device=DEV).index_fill_(
            0, torch.tensor(v, device=DEV), True) for k, v in (cons or {}).items()}
        e1 = torch.arange(int(self.off[s]), int(self.off[s + 1]), device=DEV)
        u, r1 = self.cols[e1], self.rels[e1]
        p3 = torch.arange(int(self.roff[t]), int(self.roff[t + 1]), device=DEV)
        v, r3 = self.rsrc[p3], self.rels[self.rorder[p3]]
        ok1, ok3 = (u != s) & (u != t), (v != s) & (v != t)
        if cons:
            vt = self.A["vt"].to(torch.int64)
            ok1 &= allow["rel1"][r1] & allow["types_u"][vt[u]]
            ok3 &= allow["rel3"][r3] & allow["types_v"][vt[v]]
        u, r1, v, r3 = u[ok1], r1[ok1], v[ok3], r3[ok3]
        out = torch.zeros(K, dtype=torch.float64, device=DEV)
        if not u.numel() or not v.numel():
            return out, 0
        w1 = self.weight(torch.full_like(u, s), r1, u)
        w3 = self.weight(v, r3, torch.full_like(v, t))
        ud, ui, uc = torch.unique_consecutive(u, return_inverse=True, return_counts=True)
        vd, vi, vc = torch.unique_consecutive(v, return_inverse=True, return_counts=True)
        lowest = torch.finfo(torch.float64).min
        b1 = torch.full((ud.numel(),), lowest, dtype=torch.float64, device=DEV).scatter_reduce(0, ui, w1, "amax")
        b3 = torch.full((vd.numel(),), lowest, dtype=torch.float64, device=DEV).scatter_reduce(0, vi, w3, "amax")
        mark = torch.full((self.n,), -1, dtype=torch.int64, device=DEV)
        mark[vd] = torch.arange(vd.numel(), device=DEV)
        own, e2 = self.rows_of(ud)
        at = mark[self.cols[e2]]
        keep = at >= 0
        if cons:
            keep &= allow["rel2"][self.rels[e2]]
        own, e2, at = own[keep], e2[keep], at[keep]
        if not own.numel():
            return out, 0
        w2 = self.weight(ud[own], self.rels[e2], vd[at])
        best = b1[own] + w2 + b3[at]
        kth = torch.topk(best, min(K, best.numel())).values[-1]
        keep = best >= kth - 1e-9
        own, at, w2 = own[keep], at[keep], w2[keep]
        # the parallel edges of the kept hits
        combos = uc[own] * vc[at]
        hit = torch.repeat_interleave(torch.arange(own.numel(), device=DEV), combos)
        pos = torch.arange(hit.numel(), device=DEV) - (torch.cumsum(combos, 0) - combos)[hit]
        i = (torch.cumsum(uc, 0) - uc)[own[hit]] + pos // vc[at[hit]]
        j = (torch.cumsum(vc, 0) - vc)[at[hit]] + pos % vc[at[hit]]
        top = torch.topk(w1[i] + w2[hit] + w3[j], min(K, hit.numel())).values
        out[:top.numel()] = top
        return out, top.numel()

    def beam(self, S, T, H, K):
        """Scores of the K best results of the per-path beam search, per query."""
        q = torch.arange(S.numel(), device=DEV)
        trail = [S]
        score = torch.zeros(S.numel(), dtype=torch.float64, device=DEV)
        res_q, res_s = [], []
        for level in range(H):
            x = trail[-1]
            own, e = self.rows_of(x)
            y = self.cols[e]
            ok = torch.ones_like(own, dtype=torch.bool)
            for old in trail:
                ok &= old[own] != y
            hit = y == T[q[own]]
            if level + 1 == H:
                ok &= hit
            own, e, y, hit = own[ok], e[ok], y[ok], hit[ok]
            s = score[own] + self.weight(x[own], self.rels[e], y)
            # a held path's own K best results and K best extensions
            for part, results in ((hit, True), (~hit, False)):
                po, ps, py = own[part], s[part], y[part]
                order = torch.argsort(ps, descending=True, stable=True)
                order = order[torch.argsort(po[order], stable=True)]
                po, ps, py = po[order], ps[order], py[order]
                cnt = torch.bincount(po, minlength=x.numel())
                rank = torch.arange(po.numel(), device=DEV) - (torch.cumsum(cnt, 0) - cnt)[po]
                po, ps, py = po[rank < K], ps[rank < K], py[rank < K]
                if results:
                    res_q.append(q[po])
                    res_s.append(ps)
                else:
                    kept = (po, ps, py)
            po, score, py = kept
            q, trail = q[po], [old[po] for old in trail] + [py]
        rq, rs = torch.cat(res_q), torch.cat(res_s)
        out = torch.zeros((S.numel(), K), dtype=torch.float64, device=DEV)
        for i in range(S.numel()):
            top = torch.sort(rs[rq == i], descending=True).values[:K]
            out[i, :top.numel()] = top
        return out


def exact(case, seed):
    c = case
    f, K = c["family"], c["K"]
    if f in ("batch", "load") and c["nq"] > 1024:
        return None  # minutes
    A = _arrays(c, seed)
    x = _Exact(c, A)
    if f in ("one", "batch", "noalloc", "load"):
        x.reverse()
        S, T = A["S"].tolist(), A["T"].tolist()
        got = [x.paths(s, t, K, _constraints(c) if c["constrained"] else None) for s, t in zip(S, T)]
        if f == "one":
            return {"score": got[0][0][:got[0][1]], "u": None, "v": None, "r1": None, "r2": None, "r3": None}
        return {"score": torch.stack([g[0] for g in got]), "ids": None, "n": None}
    if f == "tail":
        cand = A["vemb"] if c["cand"] < 0 else A["vemb"][A["vt"] == c["cand"]]
        h, w = A["vemb"][A["S"].to(torch.int64)].double(), A["remb"][A["Rq"].to(torch.int64)].double()
        out = torch.zeros((c["nq"], K), dtype=torch.float64, device=DEV)
        cand = cand.double()
        s = 1.0 - torch.cdist(h + w, cand, p=1.0) if c["score"] == "transe" else (h * w) @ cand.T
        top = torch.topk(s, min(K, s.shape[1]), dim=1).values
        out[:, :top.shape[1]] = top
        return {"score": out, "ids": None, "n": None}
    if f == "beam":
        return {"score": x.beam(A["S"].to(torch.int64), A["T"].to(torch.int64), c["H"], K), "ids": None, "n": None}
    if f == "edges":
        if c["rows"]:
            return {"w": x.weight(A["src"].to(torch.int64), A["rq"].to(torch.int64), A["dst"].to(torch.int64))}
        own, e = x.rows_of(torch.arange(c["n"], device=DEV))
        return {"w": x.weight(own, x.rels[e], x.cols[e])}
    # mlp: y = w2 . relu(W1 x + b1) + b2, mean squared error, one Adam step
    m, p = c["rows"], A["params"].double()
    half = torch.zeros((c["n"], 128), dtype=torch.bfloat16, device=DEV)
    w = min(128, c["d"])
    half[:, :w] = A["vemb"][:, :w].to(torch.bfloat16)
    X = torch.cat([half[A["va"].to(torch.int64)], half[A["vb"].to(torch.int64)]], 1).double()
    W1 = A["params"][:65536].to(torch.bfloat16).double().view(256, 256)
    b1, w2, b2 = p[65536:65792], p[65792:66048], p[66048]
    z = X @ W1.T + b1
    a = z.clamp(min=0)
    y = a @ w2 + b2
    err = y - A["target"].double()
    dy = 2.0 * err / m
    dz = (z > 0) * dy[:, None] * w2
    g = torch.cat([(dz.T @ X).reshape(-1), dz.sum(0), a.T @ dy, dy.sum().reshape(1)])
    step, lr, be1, be2 = 101, 1e-3, 0.9, 0.999
    m1 = be1 * A["m1"].double() + (1 - be1) * g
    m2 = be2 * A["m2"].double() + (1 - be2) * g * g
    new = p - lr * (m1 / (1 - be1 ** step)) / ((m2 / (1 - be2 ** step)).sqrt() + 1e-8)
    return {"X": X, "y": y, "z1": z, "grads": g, "loss": (err * err).mean().reshape(1), "params": new, "m1": m1,
            "m2": m2, "W1": new[:65536]}
