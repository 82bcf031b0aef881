"""Launches of the register kernel that a default handle's few-step calls leave to
the streaming kernel: one, two and three steps, and the first launch after one
that timed out.  A test hook or a chosen tile keeps these calls on the systolic
kernel.
"""
import numpy as np
import pytest
import torch

from helpers import bits_equal
from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl
from test_storage16 import REG_TILES, UNIT, _oracle16

pytestmark = pytest.mark.gpu
DT = wl.DT_DEFAULT


def run(shape, calls, scheme="systolic", source=None, order=None, **kw):
    sim = fdtd.Sim(shape, wl.random_eps(shape, 6), DT, scheme=scheme, max_source_steps=64, **kw)
    sim.write_fields(torch.as_tensor(wl.random_fields(shape, 6)).cuda())
    if source:
        sim.add_source(*source)
    if order is not None:  # the hook keeps short calls on the systolic kernel
        sim.debug_set(fdtd.DEBUG_ORDER, 0, order)
    for n in calls:
        sim.step(n)
    out, launches = sim.read_fields().cpu(), sim.launch_count
    sim.close()
    return out, launches


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("scales", [(0.5,) * 6, (1.0, 2.0, 0.5, 1.0, 1.0, 0.25)], ids=["uniform", "per-component"])
@pytest.mark.parametrize("tile", REG_TILES)
def test_16_bit_first_steps_match_oracle_emulation(cuda_device, storage, scales, tile):
    """The bounds of the same test of a default handle: a value differs from the emulation by a rounding at most."""
    shape = (24, 28, 40)
    src = (2, 20, 14, 12, wl.sine_source(3, DT))
    u, scales = UNIT[storage], np.array(scales)
    floor = scales[:, None, None, None] * (2.0 ** -24 if storage == "f16" else 0.0)
    for steps in (1, 3):
        ref = _oracle16(shape, wl.random_eps(shape, 6), wl.random_fields(shape, 6), steps, storage, scales, [src])
        got, launches = run(shape, [steps], source=src, order=2, storage=storage, field_scale=scales, tile=tile)
        got = got.numpy().astype(np.float64)
        assert launches == 1
        diff = np.abs(got - ref)
        ulp = 2.0 * u * np.maximum(np.abs(ref), np.abs(got)) + floor
        frac = (diff > 0).mean()
        if steps == 1:
            assert (diff[3:] <= ulp[3:]).all()
            assert (diff[:3] <= ulp[:3] + 4.0 * DT * max(ulp[c].max() for c in range(3, 6))).all()
            assert frac <= 5e-3
        else:
            for c in range(6):
                assert diff[c].max() <= 64.0 * u * np.abs(ref[c]).max() + floor[c].max()
            assert frac <= 5e-2


@pytest.mark.parametrize("kw", [{"tile": t} for t in sorted(fdtd.TILES)] + [
    {"tile": "31x15x12", "storage": "f16"}, {"tile": "31x15x8", "storage": "bf16"}, {"cluster": (2, 1, 1)},
    {"tile": "31x15x12", "boundary": "graded", "absorber": (3, 0.5, 3)}])
def test_launches_of_one_and_two_steps(cuda_device, kw):
    shape = (30, 45, 70)
    src = (2, 35, 22, 15, wl.sine_source(64, DT))
    plain = {k: v for k, v in kw.items() if k not in ("tile", "cluster")}
    for steps in (11, 12):
        ref, _ = run(shape, [steps], "naive", src, **plain)
        got, launches = run(shape, [steps], "systolic", src, steps_per_launch=5, **kw)
        assert launches == 3 and bits_equal(ref, got)  # 5 + 5 + 1 and 5 + 5 + 2
    got, launches = run(shape, [1, 2, 1], "systolic", src, order=2, **kw)
    assert launches == 3 and bits_equal(run(shape, [4], "naive", src, **plain)[0], got)


@pytest.mark.parametrize("kw", [{}] + [{"tile": t} for t in sorted(fdtd.TILES)])
def test_launch_after_a_timeout(cuda_device, kw):
    """The flags, the epoch and the tickets that a failed launch leaves behind don't reach the next one."""
    shape = (40, 40, 40)
    f0 = torch.as_tensor(wl.random_fields(shape, 6)).cuda()
    sim = fdtd.Sim(shape, wl.random_eps(shape, 6), DT, timeout_s=0.2, **kw)
    sim.write_fields(f0)
    sim.debug_set(fdtd.DEBUG_SKIP_PUBLISH, 3)
    sim.step(40)
    with pytest.raises(fdtd.FdtdError) as e:
        sim.sync()
    assert e.value.status == fdtd.FDTD_ERR_TIMEOUT
    sim.debug_set(fdtd.DEBUG_NONE)
    sim.write_fields(f0)
    sim.step(40)  # past the few steps that the streaming kernel takes
    got = sim.read_fields().cpu()
    sim.close()
    assert bits_equal(run(shape, [40], "naive")[0], got)
