"""Queries with fewer than K paths and many middle edges: no threshold can be found, so
one block gives the query up after the edges it may read alone (2^18 and 2^14 per
query of the batch) and the join reads them once, with its own first pass of 2^15
edges.  The lists are the oracle's."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def two_fans(rng, us, deg, vs, indeg, joins):
    """s=0 -> us vertices of out-degree deg; vs vertices of in-degree indeg -> t=1; `joins` edges between the fans."""
    U = 2 + np.arange(us)
    V = 2 + us + np.arange(vs)
    lo = 2 + us + vs
    n = lo + max(4 * deg, indeg)
    src = [np.zeros(us, np.int64), V, np.repeat(U, deg)]
    dst = [U, np.ones(vs, np.int64), (rng.integers(0, 2 * deg, us * deg) * 2 + lo)]
    src.append(np.tile(np.arange(indeg) + lo, vs))
    dst.append(np.repeat(V, indeg))
    src.append(rng.choice(U, joins))
    dst.append(rng.choice(V, joins))
    src, dst = np.concatenate(src), np.concatenate(dst)
    off, cols, rels = synth.canonicalize(n, 1, src, np.zeros(len(src), np.int64), dst)
    return synth.KG(n=n, R=1, n_types=1, offsets=off, cols=cols, rels=rels, vtypes=np.zeros(n, np.uint8),
                    vemb=(rng.standard_normal((n, 8)) * 0.3).astype(np.float32),
                    remb=(rng.standard_normal((1, 8)) * 0.3).astype(np.float32))


@pytest.mark.parametrize("joins", [0, 6])
@pytest.mark.parametrize("nq", [1, 3])
def test_a_query_without_a_threshold_is_read_once(joins, nq):
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng([joins, nq])
    g = two_fans(rng, 4000, 250, 5, 220_000, joins)
    od, ind = np.diff(g.offsets), np.bincount(g.cols, minlength=g.n)
    s_f = int(od[g.cols[: od[0]]].sum())
    s_b = int(ind[g.src_of_edges()[g.cols == 1]].sum())
    s_near = min(s_f, s_b)
    assert s_near > 600_000
    S, T = np.zeros(nq, np.uint32), np.ones(nq, np.uint32)
    want, n_want = oracle.topk_paths_batch(g, S[:1], T[:1], 50)
    G = mhr.load_kg(g)
    out, n_out, st = mhr.mhr_topk_paths_batched(G, S, T, 50, opts={"prune": 1, "order": 1}, with_stats=True)
    G.close()
    for q in range(nq):
        assert n_out[q] == n_want[0] and out[q][: n_out[q]].tobytes() == want[0][: n_want[0]].tobytes()
    assert st["edges_scanned"] <= nq * (s_near + (1 << 18) + (nq << 14) + (1 << 15))
