"""Error bounds of a loaded graph against the same formulas on norms summed in fp64 by
NumPy.  Both sums have a relative error below 4 d 2^-53 (1e-12 at these lengths)."""

import numpy as np
import pytest

from tests._graphs import random_kg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype", [(1, "f32"), (31, "f32"), (33, "f32"), (128, "f32"), (300, "f32"), (64, "bf16")])
@pytest.mark.parametrize("kind", ["plain", "unit_rows", "tiny", "one_row", "few_edges"])
def test_bounds_from_fp64_norms(d, dtype, kind):
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng([d, len(kind)])
    g = random_kg(rng, 3000, 20 if kind == "few_edges" else 9000, 40, d, dtype=dtype)
    if dtype == "f32" and kind == "unit_rows":
        g.vemb /= np.linalg.norm(g.vemb, axis=1, keepdims=True)
    elif dtype == "f32" and kind == "tiny":
        g.vemb *= np.float32(3e-23)
    elif dtype == "f32" and kind == "one_row":
        g.vemb[2990] *= np.float32(50)
    ve, re_ = np.abs(g.vemb_f32().astype(np.float64)), np.abs(g.remb_f32().astype(np.float64))
    gamma, u = 2.5, 2.0 ** -24

    def gam(k, u):
        return k * u / (1 - k * u)

    N = 2 * ve.sum(1).max() + re_.sum(1).max()
    M = re_.max() * (ve * ve).sum(1).max()
    for fn, e32, e64 in (("transe", gam(d + 4, u) * (N + gamma + 1), gam(d + 4, 2.0 ** -53) * (N + gamma + 1)),
                         ("distmult", gam(d + 3, u) * M, gam(d + 3, 2.0 ** -53) * M)):
        G = mhr.load_kg(g, score_fn=fn, gamma=gamma)
        info = mhr.mhr_graph_get_info(G)
        G.close()
        assert info["eps32_edge"] == pytest.approx(e32, rel=1e-12)
        assert info["eps64_edge"] == pytest.approx(e64, rel=1e-12)
        wmax = gamma + N if fn == "transe" else M
        path = 3 * (e32 + e64) + (gam(2, u) + gam(2, 2.0 ** -53)) * 3 * (wmax + e32 + e64)
        assert info["err_path"] == pytest.approx(path * (1 + 1e-6), rel=1e-12)
