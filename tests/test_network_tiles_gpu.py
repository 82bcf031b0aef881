"""The network's training kernels at the edges of their 32-sample tiles.

Bounds: a value of the forward pass is two dot products of at most 81 packed
roundings and a few more (2^-24 each), so 1e-5 of the largest output; a
gradient element is a sum whose chain has at most 128 roundings (32 samples
a tile, a thread's share of the partials, the activations before it), about
8e-6 of the sum of its terms' magnitudes, which random signs leave at least
a tenth of: 1e-4 relative L2 per parameter block.
"""
import numpy as np
import pytest
import torch

from oracle import mlp
from paper_2502_20610_gb300 import fdtd

pytestmark = pytest.mark.gpu
BLOCKS = {"W1": (0, 20736), "b1": (20736, 20800), "W2": (20800, 24896), "b2": (24896, 24960), "W3": (24960, 25344),
          "b3": (25344, 25350)}


def off_by_one_float(a):
    """A CUDA float32 copy of `a` that starts 4 bytes past a 16-byte boundary."""
    t = torch.empty(a.size + 5, dtype=torch.float32, device="cuda")
    v = t[1:1 + a.size].view(a.shape) if t.data_ptr() % 16 == 0 else t[:a.size].view(a.shape)
    v.copy_(torch.tensor(a, dtype=torch.float32))
    return v


# one sample, one short of a tile, a tile, one over, several tiles a CTA (152
# CTAs at most) with a ragged last one
@pytest.mark.parametrize("n", [1, 31, 32, 33, 152 * 32 + 1, 10000])
@pytest.mark.parametrize("aligned", [True, False])
def test_gradient_and_forward(cuda_device, n, aligned):
    theta = mlp.init_params(11)
    rng = np.random.default_rng(n)
    x, y = rng.standard_normal((n, mlp.N_IN)), rng.standard_normal((n, mlp.N_OUT))
    put = (lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")) if aligned else off_by_one_float
    p, xd, yd = put(theta), put(x), put(y)
    assert aligned or xd.data_ptr() % 16
    ref, _ = mlp.forward(theta, x)
    got = fdtd.mlp_forward(p, xd, batch=256).cpu().numpy()
    assert np.abs(got - ref).max() < 1e-5 * max(1.0, np.abs(ref).max())
    g_ref, l_ref = mlp.grad(theta, x, y), mlp.loss(theta, x, y)
    g, loss = fdtd.mlp_grad(p, xd, yd)
    g = g.cpu().numpy().astype(np.float64)
    assert abs(loss - l_ref) <= 1e-5 * l_ref
    for name, (a, b) in BLOCKS.items():
        assert np.linalg.norm(g[a:b] - g_ref[a:b]) <= 1e-4 * np.linalg.norm(g_ref[a:b]) + 1e-9, name
    again, _ = fdtd.mlp_grad(p, xd, yd)
    assert torch.equal(again.cpu(), torch.tensor(g, dtype=torch.float32))  # the sums have a fixed order


def test_an_infinite_input_saturates_its_sample_only(cuda_device):
    theta = mlp.init_params(12)
    x = np.random.default_rng(13).standard_normal((40, mlp.N_IN)).astype(np.float32)
    x[7, 100] = np.inf
    got = fdtd.mlp_forward(torch.tensor(theta, dtype=torch.float32, device="cuda"), torch.tensor(x, device="cuda")).cpu()
    ref, _ = mlp.forward(theta.astype(np.float32).astype(np.float64), x.astype(np.float64))
    assert np.isfinite(ref).all()
    assert np.abs(got.numpy() - ref).max() < 1e-5 * max(1.0, np.abs(ref).max())


def test_training_is_the_same_minibatches_in_the_same_order(cuda_device):
    """Two epochs over three minibatches and a rest equal one run repeated."""
    rng = np.random.default_rng(14)
    x = torch.tensor(rng.standard_normal((3 * 70 + 9, mlp.N_IN)), dtype=torch.float32, device="cuda")
    y = torch.tensor(rng.standard_normal((3 * 70 + 9, mlp.N_OUT)), dtype=torch.float32, device="cuda")
    out = []
    for _ in range(2):
        p = torch.tensor(mlp.init_params(15), dtype=torch.float32, device="cuda")
        out.append((fdtd.mlp_train(p, x, y, epochs=3, batch=70, seed=5), p.cpu()))
    assert out[0][0] == out[1][0] and torch.equal(out[0][1], out[1][1])
