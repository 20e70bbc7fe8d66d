"""fp64 scores of returned paths where the integer route of the exact TransE
weights ends: coordinates that are no multiple of its unit (tiny values beside
large ones, subnormals), rows that are not a multiple of four, of 32 or of 128,
very small and very large tables, and bands on both sides of the final merge's
pairwise limit.  Bit-identical to the oracle."""

import numpy as np
import pytest

import oracle
import synth
from tests._graphs import random_kg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype", [(1, "f32"), (6, "f32"), (31, "f32"), (33, "f32"), (128, "f32"), (130, "f32"),
                                     (300, "f32"), (8, "bf16"), (129, "bf16"), (256, "bf16")])
@pytest.mark.parametrize("kind", ["plain", "tiny_values", "small", "large"])
def test_scores_over_the_integer_route(d, dtype, kind):
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng([d, len(kind)])
    g = random_kg(rng, 150, 4000, 4, d)
    for tab in (g.vemb, g.remb):
        if kind == "tiny_values":
            m = rng.random(tab.shape)
            tab[m < 0.2] *= np.float32(1e-7)
            tab[(m >= 0.2) & (m < 0.25)] = np.float32(1e-41)
        elif kind == "small":
            tab *= np.float32(1e-20)
        elif kind == "large":
            tab *= np.float32(1e4)
    if dtype == "bf16":
        g.vemb, g.remb, g.dtype = synth.to_bf16_bits(g.vemb), synth.to_bf16_bits(g.remb), "bf16"
    S = rng.integers(0, g.n, 6).astype(np.uint32)
    T = rng.integers(0, g.n, 6).astype(np.uint32)
    T[T == S] = (T[T == S] + 1) % g.n
    for fn in ("transe", "distmult"):
        for K in (7, 300):
            want, n_want = oracle.topk_paths_batch(g, S, T, K, fn=fn)
            G = mhr.load_kg(g, score_fn=fn)
            out, n_out = mhr.mhr_topk_paths_batched(G, S, T, K)
            G.close()
            assert np.array_equal(n_out, n_want)
            for q in range(len(S)):
                assert out[q][: n_out[q]].tobytes() == want[q][: n_want[q]].tobytes(), (fn, K, q)


@pytest.mark.parametrize("K", [200, 256, 257, 600, 1024])
def test_bands_around_the_pairwise_limit(K):
    """Dyadic coordinates: many equal scores, so bands reach past K and past 512 entries."""
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng(K)
    g = random_kg(rng, 300, 20000, 2, 4, dyadic=True)
    S = rng.integers(0, g.n, 10).astype(np.uint32)
    T = ((S + 1 + rng.integers(0, g.n - 1, 10)) % g.n).astype(np.uint32)
    want, n_want = oracle.topk_paths_batch(g, S, T, K)
    G = mhr.load_kg(g)
    out, n_out = mhr.mhr_topk_paths_batched(G, S, T, K)
    G.close()
    assert np.array_equal(n_out, n_want)
    for q in range(len(S)):
        assert out[q][: n_out[q]].tobytes() == want[q][: n_want[q]].tobytes(), q
