"""The naive schedule on thin grids: one cooperative launch a call or two kernels a step by
an estimate of both, the same bits as the systolic kernel either way.
"""
import pytest
import torch

from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def stepped(shape, **kw):
    sim = fdtd.Sim(shape, 3.0, wl.DT_DEFAULT, **kw)
    sim.write_fields(torch.as_tensor(wl.random_fields(shape, 5, zero_pec_walls=False)).cuda())
    sim.step(20)
    out, launches = sim.read_fields(), sim.launch_count
    sim.close()
    return out.view(torch.int32), launches


# nz, ny, nx: sheets and needles along each axis, far from where the estimates meet
@pytest.mark.parametrize("shape,storage,launches", [
    ((1, 1000, 1000), "f32", 40), ((1, 700, 700), "f16", 40), ((4, 700, 700), "f32", 40), ((9, 700, 700), "f16", 40),
    ((450, 450, 1), "f32", 40), ((1, 20000, 1), "f32", 40),
    ((2, 60, 60), "f32", 1), ((5, 150, 150), "f16", 1), ((150, 150, 5), "f32", 1), ((600, 2, 600), "f32", 1),
    ((1, 1, 5000), "f32", 1), ((5000, 1, 1), "f16", 1), ((16, 64, 64), "f32", 1), ((40, 40, 12), "f16", 1)])
def test_form_and_bits(cuda_device, shape, storage, launches):
    naive, n = stepped(shape, scheme="naive", storage=storage)
    assert n == launches
    systolic, _ = stepped(shape, scheme="systolic", storage=storage, tile="31x15x12")
    assert torch.equal(naive, systolic)


def form_of_a_call(shape, steps):
    """(fields after the call, did the cooperative kernel run it).  Its grid barrier counts generations in word 20 of the
    handle's control words, the last 256 bytes of the workspace."""
    sim = fdtd.Sim(shape, 3.0, wl.DT_DEFAULT)
    sim.write_fields(torch.as_tensor(wl.random_fields(shape, 5, zero_pec_walls=False)).cuda())
    sim.step(steps)
    out = sim.read_fields().view(torch.int32)
    generations = int(sim.workspace[-256:].view(torch.int32)[20])
    sim.close()
    assert generations in (0, 2 * steps - 1)
    return out, generations > 0


# sheets across x, whose rows leave most lanes of a warp idle, and grids that fill them
@pytest.mark.parametrize("shape,steps,streaming", [
    ((450, 450, 1), 20, False), ((700, 700, 3), 12, False), ((700, 700, 3), 3, True), ((300, 300, 33), 18, False),
    ((300, 300, 33), 5, True), ((2000, 10, 10), 60, True), ((300, 40, 40), 18, True), ((64, 64, 64), 8, True),
    ((64, 64, 64), 40, False), ((500, 100, 20), 25, True)])
def test_which_calls_of_few_steps_stream(cuda_device, shape, steps, streaming):
    out, streamed = form_of_a_call(shape, steps)
    assert streamed == streaming
    sim = fdtd.Sim(shape, 3.0, wl.DT_DEFAULT, scheme="naive")
    sim.write_fields(torch.as_tensor(wl.random_fields(shape, 5, zero_pec_walls=False)).cuda())
    sim.step(steps)
    assert torch.equal(out, sim.read_fields().view(torch.int32))
    sim.close()
