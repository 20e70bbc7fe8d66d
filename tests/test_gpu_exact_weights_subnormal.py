"""Exact TransE weights of tables whose coordinates are all subnormal or next to it:
the integer route's unit is never finer than 2^-149, the unit of binary32 itself.
Edge scores, path lists, tail lists, beams and the no-allocation query, bit-identical
to the oracle; gamma 0 lets the tiny sums show."""

import numpy as np
import pytest

import oracle
from tests._graphs import random_kg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-37, 1e-39, 2.3e-41, 1e-44])
@pytest.mark.parametrize("d", [16, 64, 100])
def test_tables_of_the_smallest_numbers(scale, d):
    import paper_2406_07727_gb300 as mhr
    import torch
    rng = np.random.default_rng([d, int(-np.log10(scale))])
    g = random_kg(rng, 120, 3000, 3, d)
    g.vemb *= np.float32(scale)
    g.remb *= np.float32(scale)
    S = rng.integers(0, g.n, 5).astype(np.uint32)
    T = ((S + 1 + rng.integers(0, g.n - 1, 5)) % g.n).astype(np.uint32)
    Rq = rng.integers(0, g.R, 5).astype(np.uint16)
    K = 20
    G = mhr.load_kg(g, gamma=0.0)
    w = mhr.mhr_edge_scores(G, precision=2)
    assert w.tobytes() == oracle.edge_weights(g, g.src_of_edges(), g.rels, g.cols, gamma=0.0).tobytes()
    want, n_want = oracle.topk_paths_batch(g, S, T, K, gamma=0.0)
    out, n_out = mhr.mhr_topk_paths_batched(G, S, T, K)
    assert np.array_equal(n_out, n_want)
    tails, n_tails = mhr.mhr_tail_topk(G, S, Rq, K)
    want_t, n_want_t = oracle.tail_topk(g, S, Rq, K, gamma=0.0)
    beams, n_beams = mhr.mhr_beam_paths(G, S, T, 3, 5)
    want_b, n_want_b = oracle.beam_paths_batch(g, S, T, 3, 5, gamma=0.0)
    assert np.array_equal(n_tails, n_want_t) and np.array_equal(n_beams, n_want_b)
    buf = torch.zeros((1, K * 24), dtype=torch.uint8, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    for q in range(len(S)):
        k = int(n_want[q])
        assert out[q][:k].tobytes() == want[q][:k].tobytes(), q
        mhr.mhr_topk_paths_noalloc(G, int(S[q]), int(T[q]), K, buf, cnt)
        torch.cuda.synchronize()
        assert int(cnt[0]) == k and mhr.paths_from_device(buf, K)[0][:k].tobytes() == want[q][:k].tobytes(), q
        assert tails["score"][q][: n_tails[q]].tobytes() == want_t["score"][q][: n_tails[q]].tobytes(), q
        assert beams["score"][q][: n_beams[q]].tobytes() == want_b["score"][q][: n_beams[q]].tobytes(), q
    G.close()
