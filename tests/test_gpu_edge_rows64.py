"""fp64 edge scores over rows on both sides of the warp form's shortest, with values
the integer route does not hold, given triples and the graph's own edges, counts
that are no multiple of 32.  Bit-identical to the reference weights."""

import numpy as np
import pytest

import oracle
import synth
from tests._graphs import random_kg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype", [(1, "f32"), (15, "f32"), (16, "f32"), (31, "f32"), (32, "f32"), (33, "f32"), (50, "bf16"), (127, "f32"),
                                     (128, "f32"), (130, "f32"), (256, "bf16"), (300, "f32")])
@pytest.mark.parametrize("fn", ["transe", "distmult"])
@pytest.mark.parametrize("m", [1, 31, 33, 4999])
def test_scores64(d, dtype, fn, m):
    import torch
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng([d, m])
    g = random_kg(rng, 700, 9000, 5, d)
    p = rng.random(g.vemb.shape)
    g.vemb[p < 0.001] *= np.float32(1e-7)
    g.vemb[(p >= 0.001) & (p < 0.002)] = np.float32(1e-41)
    if dtype == "bf16":
        g.vemb, g.remb, g.dtype = synth.to_bf16_bits(g.vemb), synth.to_bf16_bits(g.remb), "bf16"
    G = mhr.load_kg(g, score_fn=fn)
    u, v = rng.integers(0, g.n, (2, m)).astype(np.uint32)
    r = rng.integers(0, g.R, m).astype(np.uint16)
    got = mhr.mhr_edge_scores(G, *[torch.from_numpy(a.view(t)).cuda() for a, t in
                                   ((u, np.int32), (r, np.int16), (v, np.int32))], precision=2)
    assert got.cpu().numpy().tobytes() == oracle.edge_weights(g, u, r, v, fn=fn).tobytes()
    every = mhr.mhr_edge_scores(G, precision=2)  # the graph's own edges, in order
    assert every.tobytes() == oracle.edge_weights(g, g.src_of_edges(), g.rels, g.cols, fn=fn).tobytes()
    G.close()
