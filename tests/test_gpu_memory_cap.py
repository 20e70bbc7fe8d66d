"""Loads under a memory cap around what the optional weight index takes: the index is
dropped, never the load.  A DistMult table with many relations and wide rows, whose
split copy is allocated after the index."""

import os

import numpy as np
import pytest

import oracle
from tests._graphs import random_kg

pytestmark = pytest.mark.gpu


def capped(mhr, g, cap, **kw):
    os.environ["MHR_GRAPH_MEMORY_CAP_BYTES"] = str(cap)
    try:
        return mhr.load_kg(g, **kw)
    finally:
        os.environ.pop("MHR_GRAPH_MEMORY_CAP_BYTES", None)


@pytest.mark.parametrize("fn", ["transe", "distmult"])
def test_every_cap_above_the_plain_graph_loads(fn):
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng(3)
    g = random_kg(rng, 200, 41000, 150, 256)
    n, E, R, d = g.n, g.E, g.R, 256
    split = 4 * R * d if fn == "distmult" else 0
    # rows and ids of both directions, types, embeddings, largest weights per vertex
    base = 2 * (8 * (n + 1) + 6 * E) + n + 4 * d * (n + R) + 8 * n + split
    plain, index = base + 8 * n * R, base + 36 * E + 80 * n + 12 * 256
    assert plain < index - 4 * R * d
    S = rng.integers(0, n, 4).astype(np.uint32)
    T = ((S + 1 + rng.integers(0, n - 1, 4)) % n).astype(np.uint32)
    want, n_want = oracle.topk_paths_batch(g, S, T, 9, fn=fn)
    with pytest.raises(mhr.MhrError) as e:
        capped(mhr, g, plain - 1, score_fn=fn)
    assert e.value.status == mhr.MHR_ENOMEM
    caps = [plain, plain + 1, index + 64, index + 4096]
    caps += [index - k for k in (1, 7, 8, 9, 16, 3072, split // 2 + 8, split - 8, split, split + 8, split + 3072) if k]
    for cap in caps:
        G = capped(mhr, g, cap, score_fn=fn)
        out, n_out = mhr.mhr_topk_paths_batched(G, S, T, 9)
        G.close()
        assert np.array_equal(n_out, n_want), cap
        for q in range(4):
            assert out[q][: n_out[q]].tobytes() == want[q][: n_want[q]].tobytes(), (cap, q)
