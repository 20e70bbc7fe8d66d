"""The autotuner times the form its candidates shape: the join, with and without a
weight index.  The tensor-core screen computes all 16 relations of every hit where the
fp32 screen computes one (a join that spends most of its time there takes over twice as
long); the threshold search, which reads neither, gave both the same time."""

import os

import numpy as np
import pytest

from tests._graphs import random_kg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("indexed", [True, False])
def test_screens_differ(indexed):
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng(12)
    g = random_kg(rng, 2000, 500_000, 16, 256)
    S = rng.integers(0, g.n, 48).astype(np.uint32)
    T = ((S + 1 + rng.integers(0, g.n - 1, 48)) % g.n).astype(np.uint32)
    if not indexed:
        os.environ["MHR_GRAPH_MEMORY_CAP_BYTES"] = str(g.E * 12 + 16 * (g.n + 1) + 9 * g.n + g.vemb.nbytes +
                                                       2 * g.remb.nbytes + 8 * g.n * g.R + 4096)
    try:
        G = mhr.load_kg(g, score_fn="distmult")
    finally:
        os.environ.pop("MHR_GRAPH_MEMORY_CAP_BYTES", None)
    bc, bt, bp, ms = mhr.mhr_autotune(G, S, T, 20, opts={"precision": -1}, chunks=(16384,), tiles=(4, 8), reps=3)
    assert bp == 0 and ms[(bp, bc, bt)] == min(ms.values())
    assert min(ms[(1, 16384, t)] for t in (4, 8)) > 1.5 * min(ms[(0, 16384, t)] for t in (4, 8)), ms
    # the time of a call that runs the join (its own counters)
    best = min(mhr.mhr_topk_paths_batched(G, S, T, 20, opts={"chunk": bc, "tile": bt}, with_stats=True)[2]["ms_device"]
               for _ in range(4))
    assert 0.6 * best < ms[(bp, bc, bt)] < 1.7 * best, (best, ms)
    G.close()
