"""The wait limit of the cooperative streaming kernel's grid barrier.

A handle's control words are the last 256 bytes of its workspace: the error word
and its details at 1 to 3, the barrier's count of arrivals at 16.  A count that
starts below zero is a barrier that never completes.
"""
import time

import pytest
import torch

from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
SHAPE = (40, 41, 42)


def sim_of(scheme, timeout_s):
    sim = fdtd.Sim(SHAPE, wl.random_eps(SHAPE, 2), wl.DT_DEFAULT, scheme=scheme, timeout_s=timeout_s)
    sim.write_fields(torch.as_tensor(wl.random_fields(SHAPE, 2)).cuda())
    return sim


def test_a_short_systolic_call_keeps_the_callers_limit(cuda_device):
    sim = sim_of("systolic", 0.1)
    sim.step(2)
    good = sim.read_fields()
    control = sim.workspace[-256:].view(torch.int32)
    assert control[1] == 0 and control[16] == 0
    control[16] = -100000
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    sim.step(2)
    with pytest.raises(fdtd.FdtdError) as e:
        sim.sync()
    took = time.perf_counter() - t0
    assert e.value.status == fdtd.FDTD_ERR_TIMEOUT
    assert 0.1 <= took < 1.0, took
    assert control[1] != 0 and control[3] == -5  # what was waited for
    with pytest.raises(fdtd.FdtdError):
        sim.step(1)
    # writing the fields clears the barrier with the error
    sim.write_fields(torch.as_tensor(wl.random_fields(SHAPE, 2)).cuda())
    sim.step(2)
    assert torch.equal(good.view(torch.int32), sim.read_fields().view(torch.int32))
    sim.close()


def test_a_naive_call_takes_any_limit(cuda_device):
    """The limit was the systolic scheme's: naive calls ran under any."""
    out = []
    for limit in (1e-9, 2.0):
        sim = sim_of("naive", limit)
        sim.step(7)
        out.append(sim.read_fields().view(torch.int32))
        sim.close()
    assert torch.equal(*out)
