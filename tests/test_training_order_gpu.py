"""Training, step by step against float64: the shuffled minibatches in the order that
the seed defines, and Adam's corrections.
"""
import numpy as np
import pytest
import torch

from oracle import mlp
from paper_2502_20610_gb300 import fdtd
from perf.cases import shuffle, twister
from test_network_tiles_gpu import off_by_one_float


def samples(n, seed):
    """Inputs of unit scale and the answers of another network: gradients point somewhere."""
    x = np.random.default_rng(seed).standard_normal((n, mlp.N_IN)).astype(np.float32)
    y, _ = mlp.forward(mlp.init_params(seed + 9), x)
    return x, y.astype(np.float32)


def train64(theta, x, y, batch, epochs, lr, seed, t=0):
    """Adam over the epochs' shuffled whole minibatches: (parameters, mean loss of the last epoch)."""
    theta, x, y = np.array(theta, np.float64), np.asarray(x, np.float64), np.asarray(y, np.float64)
    m, v = np.zeros_like(theta), np.zeros_like(theta)
    bits, order, loss = twister(seed), list(range(len(x))), 0.0
    for _ in range(epochs):
        shuffle(order, bits)
        loss = 0.0
        for k in range(len(x) // batch):
            rows = order[k * batch:(k + 1) * batch]
            loss += mlp.loss(theta, x[rows], y[rows]) / (len(x) // batch)
            g = mlp.grad(theta, x[rows], y[rows])
            t += 1
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            theta = theta - lr * (m / (1 - 0.9 ** t)) / (np.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return theta, loss


# An Adam step moves a parameter by lr times a ratio of about 1, whatever its gradient's
# size: where FP32's error (1e-5 of a gradient's typical size, see the gradient's test)
# is as large as the gradient itself, the ratio is lost altogether.  That is one
# parameter in 1e5, sqrt(1e-5) = 0.3 % of the moves' norm, and twice that for its sign: 1 %.
MOVE_TOL = 1e-2


@pytest.mark.gpu
@pytest.mark.parametrize("n,batch,epochs", [(3 * 70 + 9, 70, 3), (128, 32, 2), (257, 33, 4)])
@pytest.mark.parametrize("aligned", [True, False])
def test_training_follows_the_seeds_order(cuda_device, n, batch, epochs, aligned):
    theta = mlp.init_params(15).astype(np.float32)
    x, y = samples(n, 14)
    put = (lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")) if aligned else off_by_one_float
    p = put(theta)
    loss = fdtd.mlp_train(p, put(x), put(y), epochs=epochs, batch=batch, lr=1e-3, seed=5)
    ref, ref_loss = train64(theta, x, y, batch, epochs, 1e-3, 5)
    moved = np.linalg.norm(ref - theta)
    off = np.linalg.norm(p.cpu().numpy() - ref) / moved
    print(f"n={n} batch={batch} epochs={epochs}: {off:.1e} of the move, loss {abs(loss - ref_loss) / ref_loss:.1e}")
    assert off < MOVE_TOL and abs(loss - ref_loss) < 1e-4 * ref_loss


def test_another_order_is_told_apart():
    """What the bound above has to see: other minibatches, other rows, a bias correction one step off."""
    theta = mlp.init_params(15).astype(np.float32)
    x, y = samples(219, 14)
    ref, _ = train64(theta, x, y, 70, 3, 1e-3, 5)
    moved = np.linalg.norm(ref - theta)
    other, _ = train64(theta, x, y, 70, 3, 1e-3, 6)
    assert np.linalg.norm(other - ref) > 10 * MOVE_TOL * moved
    rows = np.random.default_rng(0).permutation(219)  # the same epochs, a sample's row mistaken for another's
    wrong, _ = train64(theta, x[rows], y[rows], 70, 3, 1e-3, 5)
    assert np.linalg.norm(wrong - ref) > 10 * MOVE_TOL * moved
    late, _ = train64(theta, x, y, 70, 3, 1e-3, 5, t=1)
    assert np.linalg.norm(late - ref) > 3 * MOVE_TOL * moved  # (a part of the first steps only)
