"""Tail prediction over the scans' row shapes: whole 16-byte vectors held by 1 to
32 lanes with and without padding, rows taken element by element (up to 512 of
any length) and longer ones; 1 to 130 queries in chunks, candidate counts around
the rows of a warp, the sampled form; values the integer route does not hold;
bands on both sides of the pairwise order.  Equal to the oracle."""

import numpy as np
import pytest

from tests._graphs import random_kg
from tests.test_gpu_tail import queries, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mhr():
    import paper_2406_07727_gb300 as m
    return m


@pytest.mark.parametrize("dtype,dims", [("f32", (1, 3, 4, 8, 15, 16, 20)), ("f32", (32, 33, 36, 63, 64, 68, 100)),
                                        ("f32", (127, 129, 132, 255, 257, 260)), ("f32", (511, 512, 513, 516)),
                                        ("bf16", (1, 7, 8, 16, 24, 32, 40, 50)), ("bf16", (100, 127, 136, 257, 264)),
                                        ("bf16", (511, 512, 515, 520))])
@pytest.mark.parametrize("fn", ["transe", "distmult"])
def test_row_shapes(mhr, dtype, dims, fn):
    rng = np.random.default_rng([dims[0], len(dtype)])
    for k, d in enumerate(dims):
        n = (37, 129, 1000, 2049)[k % 4]
        g = random_kg(rng, n, 3 * n, 5, d, dtype=dtype, scale=0.3)
        H, Rq = queries(rng, g, (1, 9, 33)[k % 3])
        run(mhr, g, H, Rq, 20, -1 if k % 2 else 1, fn)


@pytest.mark.parametrize("nq", [1, 7, 8, 9, 130])
@pytest.mark.parametrize("dtype,d", [("f32", 96), ("f32", 50), ("bf16", 72)])
def test_chunks_of_queries(mhr, nq, dtype, d):
    rng = np.random.default_rng(nq * d)
    g = random_kg(rng, 21003, 50000, 5, d, dtype=dtype, scale=0.3)
    H, Rq = queries(rng, g, nq)
    run(mhr, g, H, Rq, 30, -1, "transe")


@pytest.mark.parametrize("K", [3, 400, 512, 513])
def test_integer_route_and_band_sizes(mhr, K):
    rng = np.random.default_rng(K)
    g = random_kg(rng, 3000, 9000, 4, 40, scale=0.3)
    m = rng.random(g.vemb.shape)
    g.vemb[m < 0.01] *= np.float32(1e-7)
    g.vemb[(m >= 0.01) & (m < 0.02)] = np.float32(1e-41)
    H, Rq = queries(rng, g, 6)
    run(mhr, g, H, Rq, K, -1, "transe")
    g = random_kg(rng, 3000, 9000, 4, 4, dyadic=True)  # ties past K
    H, Rq = queries(rng, g, 6)
    run(mhr, g, H, Rq, K, -1, "transe")
    run(mhr, g, H, Rq, K, 2, "distmult")
