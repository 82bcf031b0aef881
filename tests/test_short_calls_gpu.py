"""Short calls and the naive schedule's cooperative launch, bit for bit against
the systolic kernel.

Few steps on a systolic handle (one or two where its tile was chosen), and any
call on a naive handle whose state is at most twice L2, run in one
cooperative launch with grid barriers.  Every storage, lossy cells, sources,
extents below a warp, and columns that do not divide into the launch's warps
must give the bits of one systolic launch.
"""
import numpy as np
import pytest
import torch

from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DT = wl.DT_DEFAULT


def run(shape, calls, scheme, sources, **kw):
    sim = fdtd.Sim(shape, wl.random_eps(shape, 3), DT, scheme=scheme, max_source_steps=64, **kw)
    sim.write_fields(torch.as_tensor(wl.random_fields(shape, 3, zero_pec_walls=False)).cuda())
    for s in sources:
        sim.add_source(*s)
    for n in calls:
        sim.step(n)
    out, at, launches = sim.read_fields(), sim.current_step, sim.launch_count
    sim.close()
    return out.view(torch.int32), at, launches


@pytest.mark.parametrize("shape", [(12, 13, 11), (1, 1, 50), (70, 2, 33), (5, 40, 100), (33, 47, 65), (150, 64, 70)])
@pytest.mark.parametrize("kw", [
    {}, {"storage": "f16"}, {"storage": "bf16", "field_scale": [1, 2, 0.5, 1, 4, 1]},
    {"boundary": "graded", "absorber": (3, 0.5, 3)}, {"boundary": "graded", "absorber": (3, 0.5, 3), "storage": "f16"}])
def test_bits_of_the_systolic_kernel(cuda_device, shape, kw):
    nz, ny, nx = shape
    src = [(2, nx // 2, ny // 2, nz // 2, wl.sine_source(64, DT)), (0, nx - 1, 0, nz - 1, wl.sine_source(5, DT, 7.0))]
    long, at, n = run(shape, [9], "systolic", src, tile="31x15x12", **kw)
    assert (at, n) == (9, 1)
    short, at, n = run(shape, [1, 2, 2, 1, 1, 2], "systolic", src, **kw)
    assert (at, n) == (9, 6)
    assert torch.equal(long, short)
    mixed, _, _ = run(shape, [1, 4, 2, 2], "systolic", src, tile="31x15x12", **kw)
    default, _, n = run(shape, [9], "systolic", src, **kw)
    assert n == 1 and torch.equal(long, default)
    assert torch.equal(long, mixed)
    naive, at, _ = run(shape, [5, 1, 3], "naive", src, **kw)
    assert at == 9 and torch.equal(long, naive)


@pytest.mark.parametrize("nz,launches", [(90, 1), (128, 10)])
def test_16_bit_naive_as_one_launch_or_two_kernels_a_step(cuda_device, nz, launches):
    shape = (nz, 128, 128)
    long, _, _ = run(shape, [5], "systolic", [], tile="31x15x12", storage="f16")
    naive, _, n = run(shape, [5], "naive", [], storage="f16")
    assert n == launches and torch.equal(long, naive)


def test_backward_sweep_of_a_state_beyond_l2(cuda_device):
    """Over 96 MB of state the E half-step sweeps the grid backwards."""
    shape = (150, 161, 170)
    long, _, _ = run(shape, [4], "systolic", [], tile="31x15x12")
    naive, _, launches = run(shape, [4], "naive", [])
    assert launches == 1 and torch.equal(long, naive)


def test_steps_replay_from_a_captured_graph(cuda_device):
    """The launch keeps nothing of the host's between calls."""
    shape = (30, 31, 45)
    f0 = torch.as_tensor(wl.random_fields(shape, 4)).cuda()
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        sim = fdtd.Sim(shape, 2.0, DT, scheme="naive")
        sim.write_fields(f0)
        sim.step(4)
        sim.sync()
        sim.write_fields(f0)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            sim.step(3)
        for _ in range(4):
            g.replay()
        got = sim.read_fields()
        sim.close()
    ref, _, _ = run_plain(shape, f0, 12)
    assert torch.equal(got.view(torch.int32), ref)


def run_plain(shape, f0, n):
    sim = fdtd.Sim(shape, 2.0, DT, scheme="systolic", tile="31x15x12")
    sim.write_fields(f0)
    sim.step(n)
    out = sim.read_fields().view(torch.int32)
    sim.close()
    return out, None, None
