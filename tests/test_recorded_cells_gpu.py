"""Recording against float64, row by row in the order of the draws.

A cell is three outputs of the seeded 64-bit Mersenne Twister modulo the box's widths,
drawn again until it lies in the layer.
"""
import numpy as np
import pytest
import torch

from oracle import mlp
from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl
from perf.cases import twister

pytestmark = pytest.mark.gpu
DT = wl.DT_DEFAULT


def recorded_cells(lo, hi, thickness, count, bits):
    """The next `count` drawn cells (x, y, z)."""
    w, out = [h - l for l, h in zip(lo, hi)], []
    while len(out) < count:
        c = [next(bits) % n for n in w]
        if min(min(v, n - 1 - v) for v, n in zip(c, w)) < thickness:
            out.append([l + v for l, v in zip(lo, c)])
    return out


@pytest.mark.parametrize("size,thickness", [((1, 7, 48), 1), ((48, 1, 7), 2), ((7, 7, 7), 3), ((33, 48, 5), 2), ((48, 48, 48), 4)])
def test_recorded_rows_follow_the_draws(cuda_device, size, thickness):
    """Row by row: the normalised stencil of the cell that was drawn, 0 outside the box."""
    shape, steps, per_step = (54, 52, 56), 3, 37
    lo = tuple((n - s) // 2 for n, s in zip((56, 52, 54), size))
    hi = tuple(l + s for l, s in zip(lo, size))
    f0 = torch.as_tensor(wl.random_fields(shape, 8)).cuda()
    sim = fdtd.Sim(shape, 2.0, DT)
    sim.write_fields(f0)
    x, _ = fdtd.learned_record(sim, lo, hi, thickness, steps, per_step, seed=21)
    sim.close()
    sim = fdtd.Sim(shape, 2.0, DT, scheme="naive")
    sim.write_fields(f0)
    states = [sim.read_fields().cpu().numpy()]
    for _ in range(steps):
        sim.step(1)
        states.append(sim.read_fields().cpu().numpy())
    sim.close()
    box = [s[:, lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]] for s in states]
    bits = twister(21)
    for s in range(steps):
        cells = np.array(recorded_cells(lo, hi, thickness, per_step, bits)) - np.array(lo)
        ref = mlp.stencil_inputs(box[s + 1], box[s], cells)
        ref /= np.sqrt(np.mean(ref ** 2, axis=1, keepdims=True))
        # one rounding of a product formed in float64
        assert np.abs(x[s * per_step:(s + 1) * per_step].cpu().numpy() - ref).max() <= 2.0 ** -23 * np.abs(ref).max()
