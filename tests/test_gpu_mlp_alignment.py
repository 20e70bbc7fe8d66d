"""Gradients from pre-activations at any float address: the 16-byte loads are taken
only where the array allows them.  The same values at an aligned address give the same
bits, since both routes do the same arithmetic."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 63, 65, 700])
@pytest.mark.parametrize("shift", [1, 2, 3])
def test_pre_activations_off_a_vector_boundary(n, shift):
    import torch
    import paper_2406_07727_gb300 as mhr
    rng = np.random.default_rng([n, shift])
    m = mhr.OrderingMLP(params=(rng.standard_normal(256 * 256 + 513) * 0.06).astype(np.float32))
    dev = torch.device("cuda")
    X = torch.from_numpy(rng.standard_normal((n, 256)).astype(np.float32)).to(dev).to(torch.bfloat16).view(torch.int16)
    target = torch.from_numpy(rng.standard_normal(n).astype(np.float32)).to(dev)
    z1 = torch.empty((n, 256), device=dev)
    y = mhr.mhr_mlp_forward(m, X, None, z1)
    work = torch.empty((n, 256), device=dev)

    def grads(z):
        g, loss = torch.empty(m.params.numel(), device=dev), torch.empty(1, device=dev)
        mhr.mhr_mlp_backward(m, X, target, y, z, work, g, loss)
        return torch.cat([g, loss]).cpu().numpy()

    room = torch.empty(n * 256 + 4, device=dev)
    moved = room[shift: shift + n * 256].view(n, 256)
    moved.copy_(z1)
    assert moved.data_ptr() % 16 == 4 * shift
    assert grads(moved).tobytes() == grads(z1).tobytes()
