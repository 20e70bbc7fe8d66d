"""fp32 edge weights of consecutive CSR edges where the warp's row walk can go
wrong: runs of empty rows longer than a warp, rows longer than a warp's 32
edges, edge counts around multiples of 32, and row lengths that select each
group width of the vector scorer and the generic one.  Reference: fp64 edge
weights; tolerance: the graph's proven fp32 bound."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def sparse_graph(rng, E, d, dtype):
    """Rows 0, 1 and the last few hold the edges; thousands of empty rows lie between."""
    n, R = 5000, 3
    rows = np.array([0, 1, 2, 40, 73, 74, 4990, n - 1])
    src = rng.choice(rows, 4 * E + 64, p=[.6, .1, .05, .05, .05, .05, .05, .05])
    dst = rng.integers(0, n, src.size)
    off, cols, rels = synth.canonicalize(n, R, src, rng.integers(0, R, src.size), dst)
    keep = np.sort(rng.choice(cols.size, E, replace=False))
    u = np.repeat(np.arange(n), np.diff(off))[keep]
    off = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(u, minlength=n), out=off[1:])
    ve = (rng.standard_normal((n, d)) * 0.3).astype(np.float32)
    re_ = (rng.standard_normal((R, d)) * 0.3).astype(np.float32)
    if dtype == "bf16":
        ve, re_ = synth.to_bf16_bits(ve), synth.to_bf16_bits(re_)
    return synth.KG(n=n, R=R, n_types=1, offsets=off, cols=cols[keep], rels=rels[keep],
                    vtypes=np.zeros(n, np.uint8), vemb=ve, remb=re_, dtype=dtype)


@pytest.mark.parametrize("E", [1, 31, 32, 33, 1000, 4097])
@pytest.mark.parametrize("d,dtype", [(1, "f32"), (4, "f32"), (12, "f32"), (50, "f32"), (128, "f32"), (256, "f32"),
                                     (260, "f32"), (8, "bf16"), (24, "bf16"), (128, "bf16"), (520, "bf16")])
def test_edge_weights_over_sparse_rows(E, d, dtype):
    import paper_2406_07727_gb300 as mhr
    g = sparse_graph(np.random.default_rng([E, d]), E, d, dtype)
    src = g.src_of_edges()
    for fn in ("transe", "distmult"):
        G = mhr.load_kg(g, score_fn=fn)
        info = mhr.mhr_graph_get_info(G)
        w = mhr.mhr_edge_scores(G, precision=0)
        given = mhr.mhr_edge_scores(G, src, g.rels, g.cols, precision=0)
        G.close()
        want = oracle.edge_weights(g, src, g.rels, g.cols, fn=fn)
        bound = info["eps32_edge"] + info["eps64_edge"]
        assert np.abs(w.astype(np.float64) - want).max() <= bound
        assert np.array_equal(w, given)
