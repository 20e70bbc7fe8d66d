"""The join on graphs loaded without the weight index (a memory cap that leaves no room
for it): the form that the screens, work-item sizes, scan tiles and row orders shape.
Each call's counters show that the join ran (the expansion has a time of its own)."""

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


def load_plain(mhr, g, fn="transe"):
    split = 4 * g.R * g.d if fn == "distmult" else 0
    room = 12 * g.E + 16 * (g.n + 1) + 9 * g.n + g.vemb.nbytes + g.remb.nbytes + split + 8 * g.n * g.R
    os.environ["MHR_GRAPH_MEMORY_CAP_BYTES"] = str(room + 16)
    try:
        return mhr.load_kg(g, score_fn=fn)
    finally:
        os.environ.pop("MHR_GRAPH_MEMORY_CAP_BYTES", None)


def join(mhr, G, S, T, K, opts):
    out, n_out, st = mhr.mhr_topk_paths_batched(G, S, T, K, opts=opts, with_stats=True)
    assert st["ms_expand"] > 0, "the threshold search ran"
    return out, n_out, st


def same(out, n_out, want, n_want, ctx):
    assert np.array_equal(n_out, n_want), ctx
    for q in range(len(n_out)):
        assert out[q][: n_out[q]].tobytes() == want[q][: n_want[q]].tobytes(), (ctx, q)


def queries(rng, n, nq):
    S = rng.integers(0, n, nq).astype(np.uint32)
    return S, ((S + 1 + rng.integers(0, n - 1, nq)) % n).astype(np.uint32)


@pytest.mark.parametrize("prune", [0, 1])
def test_tensor_core_screen(mhr, prune):
    rng = np.random.default_rng(51 + prune)
    for trial in range(8):
        n = int(rng.integers(20, 400))
        g = random_kg(rng, n, int(rng.integers(100, 25 * n)), int(rng.integers(1, 17)),
                      int(rng.choice([3, 8, 16, 37, 64, 256])), dtype="bf16" if trial % 3 == 0 else "f32",
                      dyadic=trial % 4 == 0)
        S, T = queries(rng, n, 16)
        K = int(rng.choice([1, 10, 100]))
        want, n_want = oracle.topk_paths_batch(g, S, T, K, fn="distmult")
        G = load_plain(mhr, g, "distmult")
        for precision in (0, 1):
            out, n_out, _ = join(mhr, G, S, T, K, {"precision": precision, "prune": prune, "order": prune})
            same(out, n_out, want, n_want, (trial, precision))
        G.close()


@pytest.mark.parametrize("prune,order", [(0, 0), (1, 0), (1, 1)])
def test_chunks_and_tiles(mhr, prune, order):
    g = synth.gen_rmat_kg(13, 6000, 120_000, 5, 3, seed=4)
    g.vemb, g.remb = synth.gen_embeddings(g.n, g.R, 16, 0.25, seed=4)
    S, T = synth.queries_edge_biased(g, 20, seed=4)
    want, n_want = oracle.topk_paths_batch(g, S, T, 60)
    G = load_plain(mhr, g)
    for chunk in (32, 64, 1024, 16384, 32768):
        for tile in (4, 8):
            opts = {"chunk": chunk, "tile": tile, "prune": prune, "order": order}
            out, n_out, _ = join(mhr, G, S, T, 60, opts)
            same(out, n_out, want, n_want, opts)
    G.close()


def test_the_screens_on_wide_rows(mhr):
    g = synth.gen_rmat_kg(14, 12_000, 300_000, 16, 3, seed=43)
    g.vemb, g.remb = synth.gen_embeddings(g.n, g.R, 256, 1 / 16, seed=43)
    S, T = synth.queries_edge_biased(g, 32, seed=43)
    want, n_want = oracle.topk_paths_batch(g, S, T, 100, fn="distmult")
    G = load_plain(mhr, g, "distmult")
    for opts in ({}, {"prune": 1, "order": 1}, {"precision": 1}, {"prune": 1, "order": 1, "precision": 1}):
        out, n_out, _ = join(mhr, G, S, T, 100, opts)
        same(out, n_out, want, n_want, opts)
    G.close()


def test_the_autotuner_keeps_results(mhr):
    g = synth.gen_rmat_kg(14, 12000, 200_000, 6, 3, seed=41)
    g.vemb, g.remb = synth.gen_embeddings(g.n, g.R, 32, 1 / 8, seed=41)
    S, T = synth.queries_edge_biased(g, 24, seed=41)
    want, n_want = oracle.topk_paths_batch(g, S, T, 30)
    G = load_plain(mhr, g)
    opts = {"prune": 1, "order": 1}
    bc, bt, bp, ms = mhr.mhr_autotune(G, S, T, 30, opts=opts, chunks=(64, 512, 2048), tiles=(4, 8), reps=2)
    assert len(ms) == 6 and bp == 0 and ms[(0, bc, bt)] == min(ms.values())
    out, n_out, _ = join(mhr, G, S, T, 30, {**opts, "chunk": bc, "tile": bt})
    same(out, n_out, want, n_want, (bc, bt))
    G.close()


@pytest.mark.parametrize("K", [50, 500])
def test_what_the_learned_order_saves(mhr, K):
    """Natural, bound and learned order of the same pruned join: identical lists, and the trained network's order
    scans fewer middle edges and scores fewer hits than the natural one."""
    g = synth.gen_rmat_kg(15, 30000, 600_000, 8, 3, seed=31)
    g.vemb, g.remb = synth.gen_embeddings(g.n, g.R, 64, 1 / 8, seed=31)
    S, T = synth.queries_edge_biased(g, 32, seed=31)
    St, Tt = synth.queries_edge_biased(g, 400, seed=31, stream=3)
    G = load_plain(mhr, g)
    model, rep = mhr.train_ordering_mlp(G, St, Tt, epochs=4, batch=2048, lr=2e-3)
    assert rep.rows > 1000 and rep.loss_last < rep.loss_first
    base, nb, _ = join(mhr, G, S, T, K, None)
    work = {}
    for name, opts in (("natural", {"prune": 1}), ("bound", {"prune": 1, "order": 1}),
                       ("learned", {"prune": 1, "order": 2, "mlp": model})):
        out, n, st = join(mhr, G, S, T, K, opts)
        same(out, n, base, nb, name)
        work[name] = (st["edges_scanned"], st["hits"])
    print("work (scanned, hits):", work)
    assert work["learned"][0] < work["natural"][0]
    assert work["learned"][1] < work["natural"][1]
    want, n_want = oracle.topk_paths_batch(g, S[:4], T[:4], K)
    same(base[:4], nb[:4], want, n_want, "oracle")
    G.close()
