"""A query whose cheaper side is not the one it was seeded from: the probe's far table
then holds the best slots of the other row (by that row's own cut) and finds a better
threshold for the scan."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def test_the_probe_after_a_change_of_side_finds_a_threshold():
    """DistMult weights that are sums of multiples of 1/64: w1 = x_u - 16, w2 = a_u + b_v, w3 = y_v + 16.  One u and
    one v stand out, so the row of s leaves all edges and the row of t about half of them."""
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng(4)
    nu, nv, deg, K = 8000, 8000, 100, 1000
    U, V = 2 + np.arange(nu), 2 + nu + np.arange(nv)
    x, a = rng.integers(0, 128, nu) / 64, rng.integers(0, 64, nu) / 64
    y, b = rng.integers(0, 1024, nv) / 64, rng.integers(0, 1024, nv) / 64
    x[0] += 10
    y[0] += 24
    mid = (rng.integers(0, nv, nu)[:, None] + 37 * np.arange(deg)) % nv  # deg distinct ones per u
    src = np.concatenate([np.zeros(nu, np.int64), V, np.repeat(U, deg)])
    dst = np.concatenate([U, np.ones(nv, np.int64), V[mid.ravel()]])
    n = 2 + nu + nv
    off, cols, rels = synth.canonicalize(n, 1, src, np.zeros(len(src), np.int64), dst)
    e = np.zeros((n, 8), np.float32)
    e[0, :2], e[1, 2:4] = (-4, 1), (4, 1)
    e[U, 0], e[U, 1], e[U, 4], e[U, 5] = 4, x, a, 1
    e[V, 2], e[V, 3], e[V, 4], e[V, 5] = 4, y, 1, b
    g = synth.KG(n=n, R=1, n_types=1, offsets=off, cols=cols, rels=rels, vtypes=np.zeros(n, np.uint8), vemb=e,
                 remb=np.ones((1, 8), np.float32))
    w2 = a[:, None] + b[mid]
    part = w2 + y[mid]  # without w1, and without the shifts, which cancel
    thr = np.sort((part + x[:, None]).ravel())[-K]
    n_t, n_s = int((part >= thr - x.max()).sum()), int((w2 + x[:, None] >= thr - y.max()).sum())
    assert n_s > 4 * n_t  # the row of t is the cheaper side
    S, T = np.zeros(1, np.uint32), np.ones(1, np.uint32)
    want, n_want = oracle.topk_paths_batch(g, S, T, K, fn="distmult")
    G = mhr.load_kg(g, score_fn="distmult")
    out, n_out, st = mhr.mhr_topk_paths_batched(G, S, T, K, opts={"prune": 1, "order": 1}, with_stats=True)
    G.close()
    assert n_out[0] == K and out[0][:K].tobytes() == want[0][:K].tobytes()
    # The probe reads the best sixteenth of the edges, nearly all of the K best paths among them, so its threshold is
    # close to the exact one: the scan keeps at most half as many paths again.  With the seed's it keeps 3 K.
    assert st["dense_queries"] == 0 and st["paths"] <= 1.5 * K, st
