"""Tail scans of rows past 512 elements: eight elements a lane at a time and a
remainder, two queries at a time and an odd one.  Bit-identical to the oracle."""

import numpy as np
import pytest

import oracle
from tests._graphs import random_kg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype", [(513, "f32"), (545, "f32"), (767, "f32"), (768, "f32"), (769, "f32"),
                                     (515, "bf16"), (1032, "bf16")])
@pytest.mark.parametrize("fn", ["transe", "distmult"])
def test_long_rows(d, dtype, fn):
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng(d)
    g = random_kg(rng, 9000, 2000, 3, d, dtype=dtype, scale=0.2)
    H = rng.integers(0, g.n, 33).astype(np.uint32)
    Rq = rng.integers(0, g.R, 33).astype(np.uint16)
    want, n_want = oracle.tail_topk(g, H, Rq, 9, fn=fn)
    G = mhr.load_kg(g, score_fn=fn)
    for nq in (1, 2, 3, 33):
        out, n_out = mhr.mhr_tail_topk(G, H[:nq], Rq[:nq], 9)
        assert np.array_equal(n_out, n_want[:nq])
        assert out["score"].tobytes() == want["score"][:nq].tobytes() and np.array_equal(out["v"], want["v"][:nq])
    G.close()
