"""The load's radix sort where its passes change form: one tile (8,192 edges) without
counts, up to 16 tiles without a scan of them, more with.  Lists over the sorted
in-edges and the weight index are the oracle's, bit for bit."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [1, 2, 8191, 8192, 8193, 24_577, 131_071, 131_072, 131_073, 140_000])
@pytest.mark.parametrize("n", [200, 70_000])
def test_edge_counts_around_the_forms(E, n):
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng([E, n])
    R = 40
    keys = np.sort(rng.choice(190 * 190 * R, min(3 * E + 400, 190 * 190 * R), replace=False))
    ids = np.sort(np.concatenate([[0, n - 1], 1 + rng.choice(n - 2, 188, replace=False)]))
    u, v, r = keys // (190 * R), keys // R % 190, keys % R
    live = np.flatnonzero(u != v)
    live = np.sort(rng.choice(live, E, replace=False))
    off, cols, rels = synth.canonicalize(n, R, ids[u[live]], r[live], ids[v[live]])
    assert cols.size == E
    ve = np.zeros((n, 4), np.float32)
    ve[ids] = rng.standard_normal((190, 4)).astype(np.float32)
    g = synth.KG(n=n, R=R, n_types=1, offsets=off, cols=cols, rels=rels, vtypes=np.zeros(n, np.uint8), vemb=ve,
                 remb=rng.standard_normal((R, 4)).astype(np.float32))
    S, T = rng.choice(ids, 5).astype(np.uint32), rng.choice(ids, 5).astype(np.uint32)
    ok = S != T
    S, T = S[ok], T[ok]
    G = mhr.load_kg(g)
    out, n_out = mhr.mhr_topk_paths_batched(G, S, T, 40)
    beams, n_beams = mhr.mhr_beam_paths(G, S, T, 3, 6)
    G.close()
    want, n_want = oracle.topk_paths_batch(g, S, T, 40)
    want_b, n_want_b = oracle.beam_paths_batch(g, S, T, 3, 6)
    assert np.array_equal(n_out, n_want) and np.array_equal(n_beams, n_want_b)
    for q in range(len(S)):
        assert out[q][: n_out[q]].tobytes() == want[q][: n_want[q]].tobytes()
        assert beams["score"][q][: n_beams[q]].tobytes() == want_b["score"][q][: n_want_b[q]].tobytes()
