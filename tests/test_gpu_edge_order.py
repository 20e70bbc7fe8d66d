"""The fp32 edge weight's order of additions: each 16-byte vector of a row is summed
by itself, element by element, and the vectors' sums (of up to 32 vectors) are added
in a tree that first joins the vectors half the width apart.  TransE, where nothing is
fused, so the same additions in NumPy give the same bits; the index, the training
labels and the edge scores all use this weight."""

import numpy as np
import pytest

from tests._graphs import random_kg

pytestmark = pytest.mark.gpu


def tree_weight(e, r, t, ev):
    """gamma 1 minus the tree sum of |e + r - t| over rows [m, d] of float32."""
    x = np.abs((e + r).astype(np.float32) - t)
    nv = x.shape[1] // ev
    width = 1
    while width < nv:
        width *= 2
    acc = np.zeros((x.shape[0], width), np.float32)
    for j in range(ev):
        acc[:, :nv] += x[:, j::ev]
    while width > 1:
        width //= 2
        acc = acc[:, :width] + acc[:, width:]
    return np.float32(1) - acc[:, 0]


@pytest.mark.parametrize("dtype,d", [("f32", 4), ("f32", 8), ("f32", 12), ("f32", 36), ("f32", 64), ("f32", 100),
                                     ("f32", 128), ("bf16", 8), ("bf16", 24), ("bf16", 128), ("bf16", 200),
                                     ("bf16", 256)])
def test_vectors_summed_by_themselves(dtype, d):
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng(d)
    g = random_kg(rng, 400, 5001, 4, d, dtype=dtype)
    ve, re_ = g.vemb_f32(), g.remb_f32()
    want = tree_weight(ve[g.src_of_edges()], re_[g.rels], ve[g.cols], 4 if dtype == "f32" else 8)
    G = mhr.load_kg(g)
    w = mhr.mhr_edge_scores(G)
    src, rel, dst = g.src_of_edges().astype(np.uint32)[:777], g.rels[:777], g.cols[:777]
    w3 = mhr.mhr_edge_scores(G, src, rel, dst)
    G.close()
    assert w.tobytes() == want.tobytes()
    assert w3.tobytes() == want[:777].tobytes()
