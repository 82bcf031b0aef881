"""The adjoint gradient on every form of the register kernel that captures the
design box: loss and gradient are the bits of the naive schedule's.
"""
import numpy as np
import pytest
import torch

from oracle import adjoint as adj
from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DT = wl.DT_DEFAULT


def problem(shape, steps, seed=3):
    """eps with a random box in it, the box's corners (x, y, z), a mode and a source below the box."""
    nz, ny, nx = shape
    lo, hi = (nx // 3, ny // 3, nz // 3), (nx // 3 + 9, ny // 3 + 7, nz // 3 + 6)
    eps = np.full(shape, 2.1)
    u = np.asarray(wl.uniform_pm1(seed, 9 * 7 * 6), np.float64).reshape(6, 7, 9)
    eps[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]] = 7.1 + 5.0 * u
    mode = np.asarray(wl.uniform_pm1(seed + 1, ny * nx)).reshape(ny, nx)
    return eps, lo, hi, mode, (2, nx // 2, ny // 2, nz // 3 - 3, wl.sine_source(steps, DT, 10.0))


def gradient(shape, steps, window, every, **kw):
    eps, lo, hi, mode, src = problem(shape, steps)
    sim = fdtd.Sim(shape, eps, DT, max_source_steps=steps, **kw)
    sim.write_fields(torch.zeros((6,) + shape, device="cuda"))
    sim.add_source(*src)
    # a history that is never stored must not be found where another run left it
    torch.cuda.empty_cache()
    dirty = torch.full((1 << 28,), float("nan"), device="cuda")
    del dirty
    loss, grad = fdtd.adjoint_gradient(sim, hi[2] + 3, torch.as_tensor(mode), window, steps, lo, hi, every)
    state = sim.read_fields()
    sim.close()
    return loss, grad, state.view(torch.int32)


# a window shorter and longer than a segment, segments that do not divide the
# steps, an odd number of tiles along x (a pair with one tile)
@pytest.mark.parametrize("shape,steps,window,every", [((26, 24, 70), 50, 12, 20), ((30, 40, 95), 40, 25, 16)])
def test_cluster_pairs(cuda_device, shape, steps, window, every):
    pair = gradient(shape, steps, window, every, cluster=(2, 1, 1))
    naive = gradient(shape, steps, window, every, scheme="naive")
    assert pair[0] == naive[0] and pair[0] > 0.0
    assert torch.equal(pair[1], naive[1]) and torch.equal(pair[2], naive[2])


def test_twelve_row_tile(cuda_device):
    """The capturing kernel of larger domains, against the float64 adjoint as well."""
    shape, steps, window, every = (26, 24, 30), 60, 25, 20
    eps, lo, hi, mode, src = problem(shape, steps)
    loss, grad, state = gradient(shape, steps, window, every, tile="31x15x12")
    naive = gradient(shape, steps, window, every, scheme="naive")
    assert loss == naive[0] and torch.equal(grad, naive[1]) and torch.equal(state, naive[2])
    obj = adj.Objective(hi[2] + 3, mode.astype(np.float64), window)
    ref_loss, ref = adj.gradient(shape, eps, np.zeros((6,) + shape), steps, [src], obj, DT, quantize=True)
    ref = ref[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]]
    # the gradient's bound of the adjoint tests: FP32 rounding over the steps
    assert abs(loss - ref_loss) <= 1e-4 * ref_loss
    assert np.linalg.norm(grad.cpu().numpy() - ref) <= 1e-4 * np.linalg.norm(ref)
