"""Device memory of a plan: the threshold search's buffers are allocated by the first
call that runs it, not by calls that only run the join, and when there is no room
for them the join answers with the same lists."""

import numpy as np
import pytest

import oracle
from tests._graphs import random_kg

pytestmark = pytest.mark.gpu


def test_search_buffers_come_with_the_search():
    import torch
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng(2)
    g = random_kg(rng, 300, 4000, 3, 8)
    nq = 700  # two blocks on every SM
    S = rng.integers(0, g.n, nq).astype(np.uint32)
    T = ((S + 1 + rng.integers(0, g.n - 1, nq)) % g.n).astype(np.uint32)
    want, n_want = oracle.topk_paths_batch(g, S, T, 5)
    spill = 2 * torch.cuda.get_device_properties(0).multi_processor_count * (15360 + 8192) * 16

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    def same(out, n_out):
        assert np.array_equal(n_out, n_want)
        for q in range(nq):
            assert out[q][: n_out[q]].tobytes() == want[q][: n_want[q]].tobytes(), q

    G = mhr.load_kg(g)
    out, n_out, _ = mhr.mhr_topk_paths_batched(G, S, T, 5, with_stats=True)  # the join's counters
    same(out, n_out)
    before = free()
    hog = torch.empty(before - (48 << 20), dtype=torch.uint8, device="cuda")  # less than either buffer takes
    assert free() < spill
    with pytest.raises(mhr.MhrError):
        mhr.mhr_topk_paths(G, 1, 1, 5)
    said = mhr.mhr_last_error()
    same(*mhr.mhr_topk_paths_batched(G, S, T, 5))
    assert mhr.mhr_last_error() == said  # no call has failed since
    del hog
    torch.cuda.empty_cache()
    before = free()
    same(*mhr.mhr_topk_paths_batched(G, S, T, 5))
    assert before - free() >= spill
    before = free()
    same(*mhr.mhr_topk_paths_batched(G, S, T, 5))
    assert before == free()
    G.close()
