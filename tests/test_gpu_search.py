"""Threshold search over the weight index at the sizes where it can go wrong:
row lengths around the ranks kept per row (4, 32, 256, 2048) and around sectors
and pieces, far rows around the seed table's capacity, one block per query with
either block size, K from 1 to the largest with candidates past the shared buffer,
queries handed back (ties) among others, constraints and partitions, and the same
graphs loaded without the index.  Every list is the oracle's, bit for bit."""

import os

import numpy as np
import pytest

import oracle
import synth
from tests._graphs import random_kg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mhr():
    import paper_2406_07727_gb300 as m
    return m


def same(out, n_out, want, n_want):
    assert np.array_equal(n_out, n_want)
    for q in range(len(n_out)):
        assert out[q][: n_out[q]].tobytes() == want[q][: n_want[q]].tobytes(), q


def layered(rng, mids, far, degs, d=8, R=3, dup=1):
    """s=0 -> mids vertices -> (row lengths degs, into `far` vertices and elsewhere) -> t=1; `dup` relations per
    outer edge."""
    n = 2 + mids + far + 4000
    U, V = np.arange(2, 2 + mids), np.arange(2 + mids, 2 + mids + far)
    src, dst, rel = [], [], []
    for r in range(dup):
        src += [np.zeros(mids, np.int64), V]
        dst += [U, np.ones(far, np.int64)]
        rel += [np.full(mids, r), np.full(far, r)]
    for u, k in zip(U, np.resize(degs, mids)):
        into = rng.choice(far + 4000, size=int(k), replace=False) + 2 + mids
        src.append(np.full(int(k), u))
        dst.append(into)
        rel.append(rng.integers(0, R, int(k)))
    off, cols, rels = synth.canonicalize(n, R, np.concatenate(src), np.concatenate(rel), np.concatenate(dst))
    ve = (rng.standard_normal((n, d)) * 0.5).astype(np.float32)
    re_ = (rng.standard_normal((R, d)) * 0.5).astype(np.float32)
    return synth.KG(n=n, R=R, n_types=1, offsets=off, cols=cols, rels=rels, vtypes=np.zeros(n, np.uint8), vemb=ve,
                    remb=re_)


@pytest.mark.parametrize("degs", [[1, 2, 3, 4, 5], [31, 32, 33, 34], [255, 256, 257, 258, 1], [2047, 2048, 2049, 2050, 7]])
@pytest.mark.parametrize("K", [1, 60, 1024])
def test_row_lengths_around_the_kept_ranks(mhr, degs, K):
    rng = np.random.default_rng([len(degs), degs[0], K])
    g = layered(rng, 24, 900, degs, dup=2)
    S, T = np.array([0], np.uint32), np.array([1], np.uint32)
    want, n_want = oracle.topk_paths_batch(g, S, T, K)
    G = mhr.load_kg(g)
    for opts in (None, {"prune": 1, "order": 0}, {"prune": 1, "order": 1}):
        out, n_out = mhr.mhr_topk_paths_batched(G, S, T, K, opts=opts)
        same(out, n_out, want, n_want)
    G.close()


@pytest.mark.parametrize("far", [1, 500, 6143, 6145, 13000])
@pytest.mark.parametrize("copies", [1, 200])
def test_far_rows_and_block_sizes(mhr, far, copies):
    rng = np.random.default_rng([far, copies])
    g = layered(rng, 300, far, [40, 3, 90], dup=1)
    S, T = np.zeros(copies, np.uint32), np.ones(copies, np.uint32)
    want, n_want = oracle.topk_paths_batch(g, S[:1], T[:1], 50)
    G = mhr.load_kg(g)
    out, n_out = mhr.mhr_topk_paths_batched(G, S, T, 50)
    G.close()
    same(out, n_out, np.repeat(want, copies, 0), np.repeat(n_want, copies))


@pytest.mark.parametrize("fn", ["transe", "distmult"])
@pytest.mark.parametrize("indexed", [True, False])
def test_with_and_without_the_index(mhr, fn, indexed):
    """A memory cap that leaves no room for the index: the join answers; the lists are the same.  Ties on part of
    the graph send some queries from the search to the join."""
    rng = np.random.default_rng(5)
    g = random_kg(rng, 500, 30000, 4, 8)
    g.vemb[:250] = 0
    g.remb[:] = 0
    S = rng.integers(0, g.n, 180).astype(np.uint32)
    T = rng.integers(0, g.n, 180).astype(np.uint32)
    S[:8], T[:8] = np.arange(8), np.arange(8)  # invalid: s == t
    base = g.E * 12 + 16 * (g.n + 1) + g.vemb.nbytes + g.remb.nbytes + 9 * g.n
    if not indexed:
        os.environ["MHR_GRAPH_MEMORY_CAP_BYTES"] = str(base + 2 * g.n * g.R * 4 + 20000)
    try:
        G = mhr.load_kg(g, score_fn=fn)
    finally:
        os.environ.pop("MHR_GRAPH_MEMORY_CAP_BYTES", None)
    ok = np.flatnonzero(S != T)
    want, n_want = oracle.topk_paths_batch(g, S[ok], T[ok], 40, fn=fn)
    for opts in (None, {"prune": 1, "order": 1}, {"prune": 1}):
        out, n_out = mhr.mhr_topk_paths_batched(G, S, T, 40, opts=opts)
        assert (n_out[S == T] == -1).all()
        same(out[ok], n_out[ok], want, n_want)
    c = {"rel1": [0, 1], "rel2": [1, 2, 3], "rel3": [0, 3], "types_u": [0, 1], "types_v": [1, 2]}
    out, n_out = mhr.mhr_topk_paths_batched(G, S[ok[:12]], T[ok[:12]], 40, opts={"constraints": c})
    for q in range(12):
        w = oracle.topk_paths_masked(g, int(S[ok[q]]), int(T[ok[q]]), 40, fn=fn, **c)
        assert n_out[q] == len(w) and out[q][: n_out[q]].tobytes() == w.tobytes()
    parts = [mhr.mhr_topk_paths_batched(G, S[ok], T[ok], 40, opts={"part_count": 3, "part_index": r}) for r in range(3)]
    merged, n_merged = mhr.mhr_merge_paths(np.stack([p for p, _ in parts]), np.stack([n for _, n in parts]), 40)
    G.close()
    same(merged, n_merged, want, n_want)
