"""Steps on a stream that owns a part of the SMs only (a green context of this process):
a cooperative grid of a CTA on every SM doesn't fit there, and the calls that would
use one run as two kernels a step.
"""
import contextlib
import ctypes

import pytest
import torch

from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def partition(sms):
    """A torch stream on at least `sms` SMs of the device, through the driver's API (its structures kept opaque)."""
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")

    def call(name, *args):
        assert getattr(cu, name)(*args) == 0, name

    whole, part = ctypes.create_string_buffer(512), ctypes.create_string_buffer(512)
    dev, groups, desc = ctypes.c_int(), ctypes.c_uint(1), ctypes.c_void_p()
    ctx, stream = ctypes.c_void_p(), ctypes.c_void_p()
    call("cuDeviceGet", ctypes.byref(dev), torch.cuda.current_device())
    call("cuDeviceGetDevResource", dev, whole, 1)  # the SMs
    call("cuDevSmResourceSplitByCount", part, ctypes.byref(groups), whole, None, 0, ctypes.c_uint(sms))
    call("cuDevResourceGenerateDesc", ctypes.byref(desc), part, 1)
    call("cuGreenCtxCreate", ctypes.byref(ctx), desc, dev, 1)  # with a default stream, which creation requires
    call("cuGreenCtxStreamCreate", ctypes.byref(stream), ctx, 1, 0)  # non-blocking
    try:
        s = torch.cuda.ExternalStream(stream.value)
        with torch.cuda.stream(s):
            yield s
        s.synchronize()
    finally:
        call("cuStreamDestroy_v2", stream)
        call("cuGreenCtxDestroy", ctx)


def stepped(shape, calls, **kw):
    sim = fdtd.Sim(shape, wl.random_eps(shape, 3), wl.DT_DEFAULT, **kw)
    sim.write_fields(torch.as_tensor(wl.random_fields(shape, 3)).cuda())
    for n in calls:
        sim.step(n)
    out, at, launches = sim.read_fields(), sim.current_step, sim.launch_count
    sim.close()
    return out.view(torch.int32), at, launches


@pytest.mark.parametrize("kw,calls,launches", [
    ({"scheme": "naive"}, [5, 2], 14), ({"scheme": "systolic"}, [1, 2, 4], 14),
    ({"scheme": "systolic", "tile": "31x15x12"}, [2, 5], 5), ({"scheme": "naive", "storage": "f16"}, [7], 14)])
def test_every_schedule_runs_on_a_part_of_the_chip(cuda_device, kw, calls, launches):
    shape = (60, 66, 70)
    whole, _, _ = stepped(shape, calls, **kw)
    with partition(16):
        part, at, n = stepped(shape, calls, **kw)
    assert at == sum(calls) and n == launches and torch.equal(whole, part)
