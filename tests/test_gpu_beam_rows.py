"""Beam search on a graph with and without its weight index: a warp per held
path on the rows sorted by weight, a CTA per path for the rest.  Rows around K
and around the steps of 32 edges, more edges into t than a warp takes or than
K, ties wider than a warp's candidate list, vertices of the path among the
best extensions.  Equal to the oracle element by element, and the same bytes
without an index."""

import numpy as np
import pytest

import oracle
from tests._graphs import random_kg
from tests.test_gpu_beam import tuples

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,E,R,d,dtype,dyadic,H,K", [
    (40, 70, 2, 8, "f32", False, 4, 3),         # rows shorter than K, vertices without edges
    (200, 6400, 1, 16, "f32", False, 3, 32),    # rows around 32 edges, K = 32
    (200, 6400, 1, 33, "bf16", False, 2, 31),
    (60, 12000, 8, 130, "f32", False, 2, 64),   # rows of 200 edges
    (14, 6000, 60, 8, "f32", False, 3, 3),      # about 33 edges into t from every vertex: more than K
    (14, 5500, 60, 5, "f32", False, 2, 40),     # on both sides of a warp's 32
    (30, 12000, 40, 4, "f32", True, 3, 5),      # ties of hundreds of edges
    (12, 900, 9, 6, "bf16", False, 5, 6),       # most extensions are on the path
    (300, 40000, 3, 4, "f32", True, 8, 1),
])
@pytest.mark.parametrize("fn", ["transe", "distmult"])
def test_rows_and_lists(monkeypatch, n, E, R, d, dtype, dyadic, H, K, fn):
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng([n, E, K])
    g = random_kg(rng, n, E, R, d, dtype=dtype, dyadic=dyadic, scale=0.3)
    S = rng.integers(0, g.n, 8).astype(np.uint32)
    T = ((S + 1 + rng.integers(0, g.n - 1, 8)) % g.n).astype(np.uint32)
    G = mhr.load_kg(g, score_fn=fn)
    out, n_out = mhr.mhr_beam_paths(G, S, T, H, K)
    small, n_small, st = mhr.mhr_beam_paths(G, S[:1], T[:1], H, K, with_stats=True)  # kept buffers of a larger call
    G.close()
    assert tuples(small[0], int(n_small[0])) == tuples(out[0], int(n_out[0])) and st["edges_scanned"] >= 0
    for q in range(len(S)):
        want = tuples(oracle.beam_paths(g, int(S[q]), int(T[q]), H, K, fn=fn), K)
        assert tuples(out[q], int(n_out[q])) == want, q
    # room for the graph and the bounds per (vertex, relation), not for the index's 36 bytes an edge
    base = g.E * 12 + 16 * (g.n + 1) + g.vemb.nbytes + g.remb.nbytes + 9 * g.n
    monkeypatch.setenv("MHR_GRAPH_MEMORY_CAP_BYTES", str(base + 8 * n * R + 4 * R * d + 1500))
    G = mhr.load_kg(g, score_fn=fn)
    plain, n_plain = mhr.mhr_beam_paths(G, S, T, H, K)
    G.close()
    assert np.array_equal(n_plain, n_out)
    for q in range(len(S)):
        assert plain[q][: n_out[q]].tobytes() == out[q][: n_out[q]].tobytes(), q
