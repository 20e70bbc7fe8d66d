"""mhr_topk_paths_noalloc on a graph with a weight index (threshold search and
finish in one block) and without one: candidate lists up to, at and past its
buffers, rows on both sides of the integer route, queries without a path, and a
call replayed from a captured graph.  Equal to the oracle byte for byte.  Sorts
last, like the other test of this entry point."""

import numpy as np
import pytest

import oracle
from tests._graphs import random_kg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,E,R,d,kind,Ks", [
    (40, 60, 2, 4, "plain", (1, 9)),                   # most queries have no path
    (300, 6000, 3, 64, "plain", (1, 31, 1024)),
    (150, 9000, 4, 33, "tiny_values", (20, 1000)),     # sums left to the fp64 route
    (200, 20000, 2, 130, "bf16", (5, 1023)),
    (300, 20000, 2, 4, "dyadic", (200, 700, 1024)),    # bands past 1,024
    (300, 20000, 2, 16, "dyadic", (990,)),
    (80, 5000, 4, 8, "zero", (3, 1024)),               # every candidate ties: the walk
    (2000, 90000, 5, 300, "plain", (50, 400)),
])
def test_index_forms(monkeypatch, n, E, R, d, kind, Ks):
    torch = pytest.importorskip("torch")
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng([n, E, d])
    g = random_kg(rng, n, E, R, d, dtype="bf16" if kind == "bf16" else "f32", dyadic=kind == "dyadic",
                  zero=kind == "zero")
    if kind == "tiny_values":
        m = rng.random(g.vemb.shape)
        g.vemb[m < 0.2] *= np.float32(1e-7)
        g.vemb[(m >= 0.2) & (m < 0.25)] = np.float32(1e-41)
    S = rng.integers(0, g.n, 5)
    T = (S + 1 + rng.integers(0, g.n - 1, 5)) % g.n
    out = torch.empty(1024 * 24, dtype=torch.uint8, device="cuda")
    cnt = torch.empty(1, dtype=torch.int32, device="cuda")

    def read():
        torch.cuda.synchronize()
        return out.cpu().numpy().view(mhr.PATH_DTYPE)[: int(cnt.item())].tobytes()

    base = g.E * 12 + 16 * (g.n + 1) + g.vemb.nbytes + g.remb.nbytes + 9 * g.n
    for fn in ("transe", "distmult"):
        for indexed in (True, False):
            if indexed:
                monkeypatch.delenv("MHR_GRAPH_MEMORY_CAP_BYTES", raising=False)
            else:  # room for the bounds per (vertex, relation), not for the index
                monkeypatch.setenv("MHR_GRAPH_MEMORY_CAP_BYTES", str(base + 8 * n * R + 4 * R * d + 1500))
            G = mhr.load_kg(g, score_fn=fn)
            for K in Ks:
                want, n_want = oracle.topk_paths_batch(g, S.astype(np.uint32), T.astype(np.uint32), K, fn=fn)
                for q in range(len(S)):
                    out.fill_(0xAB)
                    cnt.fill_(-7)
                    mhr.mhr_topk_paths_noalloc(G, int(S[q]), int(T[q]), K, out, cnt)
                    assert read() == want[q][: n_want[q]].tobytes(), (fn, indexed, K, q)
            stream = torch.cuda.Stream()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                mhr.mhr_topk_paths_noalloc(G, int(S[0]), int(T[0]), K, out, cnt, stream=stream)
            for _ in range(2):
                out.fill_(0xCD)
                cnt.fill_(-7)
                graph.replay()
                assert read() == want[0][: n_want[0]].tobytes(), (fn, indexed)
            G.close()
