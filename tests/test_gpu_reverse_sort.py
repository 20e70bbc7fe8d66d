"""Reverse adjacency built by the load's radix sort, at the edges of its tiles
(8,192 edges) and of its passes (8 bits of the vertex id each): three-hop lists
that read the in-edges of t are compared with the oracle, bit for bit."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [3, 8191, 8192, 8193, 16384, 30001])
@pytest.mark.parametrize("n", [200, 256, 257, 65536, 70_000, (1 << 24) + 9])
def test_paths_over_sorted_in_edges(E, n):
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng([E, n])
    # the edges live among 190 vertices spread over the id range, so that paths exist
    ids = np.unique(np.concatenate([[0, 1, n - 1], rng.choice(n, 187, replace=False)]))
    m = E if E < 100 else 2 * E
    src, dst = rng.choice(ids, m), rng.choice(ids, m)
    off, cols, rels = synth.canonicalize(n, 40, src, rng.integers(0, 40, m), dst)
    keep = np.sort(rng.choice(cols.size, min(E, cols.size), replace=False))
    u = np.searchsorted(off, keep, side="right") - 1
    off = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(u, minlength=n), out=off[1:])
    ve = np.zeros((n, 4), np.float32)
    ve[ids] = rng.standard_normal((ids.size, 4)).astype(np.float32)
    re_ = rng.standard_normal((40, 4)).astype(np.float32)
    g = synth.KG(n=n, R=40, n_types=1, offsets=off, cols=cols[keep], rels=rels[keep],
                 vtypes=np.zeros(n, np.uint8), vemb=ve, remb=re_)
    S, T = rng.choice(ids, 6).astype(np.uint32), rng.choice(ids, 6).astype(np.uint32)
    ok = S != T
    S, T = S[ok], T[ok]
    G = mhr.load_kg(g)
    out, n_out = mhr.mhr_topk_paths_batched(G, S, T, 30)
    G.close()
    want, n_want = oracle.topk_paths_batch(g, S, T, 30)
    assert np.array_equal(n_out, n_want)
    for q in range(len(S)):
        assert out[q][: n_out[q]].tobytes() == want[q][: n_want[q]].tobytes()
