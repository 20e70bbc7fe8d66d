"""Gradients of the ordering MLP where their rows are cut into chunks of 64 and
slices of at least 258: against the same sums in fp64, from the same
pre-activations and outputs."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 63, 64, 65, 257, 258, 259, 515, 517, 577, 2900, 9827, 30000])
def test_backward_over_rows(n):
    torch = pytest.importorskip("torch")
    import paper_2406_07727_gb300 as mhr
    import paper_2406_07727_gb300.learn  # noqa: F401
    rng = np.random.default_rng(n)
    p = (rng.standard_normal(mhr.learn.N_PARAMS) * 0.1).astype(np.float32)
    model = mhr.OrderingMLP(params=p)
    Xb = synth.to_bf16_bits(rng.standard_normal((n, 256)).astype(np.float32))
    z1 = rng.standard_normal((n, 256)).astype(np.float32)
    y, t = rng.standard_normal((2, n)).astype(np.float32)
    work = torch.full((n, 256), float("nan"), device="cuda")  # scratch of any content
    grads = torch.empty(mhr.learn.N_PARAMS, device="cuda")
    loss = torch.empty(1, device="cuda")
    args = [torch.from_numpy(a).cuda() for a in (Xb.view(np.int16), t, y, z1)]
    runs = []
    for _ in range(2):
        grads.fill_(float("nan"))
        mhr.mhr_mlp_backward(model, *args, work, grads, loss)
        runs.append(grads.cpu().numpy().copy())
    assert runs[0].tobytes() == runs[1].tobytes()
    X = synth.bf16_bits_to_f32(Xb).astype(np.float64)
    w2 = p[65792:66048].astype(np.float64)
    e = y.astype(np.float64) - t
    dy = 2 * e / n
    relu = np.maximum(z1.astype(np.float64), 0)
    dz = (z1 > 0) * dy[:, None] * w2
    # rounding of y - t, 2 / n and the two products; the split of dZ (2^-16); n additions
    # of unit roundoff 2^-22 (tensor cores) or 2^-24
    eps = 2.0 ** -24
    cases = [(runs[0][:65536].reshape(256, 256), dz.T @ X, np.abs(dz).T @ np.abs(X), 2.0 ** -16 + 4 * eps + n * 2.0 ** -22),
             (runs[0][65536:65792], dz.sum(0), np.abs(dz).sum(0), (n + 4) * eps),
             (runs[0][65792:66048], relu.T @ dy, relu.T @ np.abs(dy), (n + 4) * eps),
             (runs[0][66048], dy.sum(), np.abs(dy).sum(), (n + 3) * eps),
             (loss.item(), (e * e).sum() / n, (e * e).sum() / n, (n + 4) * eps)]
    for k, (got, want, size, tol) in enumerate(cases):
        assert np.all(np.abs(got - want) <= 1.01 * tol * size + 1e-30), k
