"""fdtd_write_fields and fdtd_read_fields on device memory (one launch for all
components) against the host path (a copy per component), bit for bit: rows
that are and are not whole groups of four values, pointers off their 16-byte
boundary, component masks, every storage; and the error word, which the
device copy looks at itself.
"""
import numpy as np
import pytest
import torch

from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DT = wl.DT_DEFAULT


@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 7), (3, 5, 8), (4, 33, 100), (2, 9, 1030), (700, 3, 4)])
@pytest.mark.parametrize("kw", [{}, {"storage": "f16"}, {"storage": "bf16", "field_scale": [1, 2, 0.5, 1, 4, 8]}])
@pytest.mark.parametrize("offset", [0, 1])
def test_device_copies_equal_host_copies(cuda_device, shape, kw, offset):
    n = int(np.prod(shape))
    f = wl.random_fields(shape, 7, zero_pec_walls=False) * np.float32(300.0)
    f[:, 0, 0, 0] = [0.0, -0.0, 1e-30, -1e-30, 7.0, -7.0]
    sim = fdtd.Sim(shape, 2.0, DT, **kw)
    sim.write_fields(f)  # host
    host = np.empty((6,) + shape, np.float32)
    sim.read_fields_ptr(0x3F, host.ctypes.data)
    src = torch.zeros(6 * n + 8, device="cuda")
    src[offset:offset + 6 * n] = torch.from_numpy(f).cuda().reshape(-1)
    sim.write_fields(np.zeros_like(f))
    sim.write_fields_ptr(src[offset:].data_ptr())
    again = np.empty((6,) + shape, np.float32)
    sim.read_fields_ptr(0x3F, again.ctypes.data)
    assert np.array_equal(host.view(np.int32), again.view(np.int32))
    for mask in (0x3F, 0x01, 0x2A, 0x34):
        comps = [c for c in range(6) if mask & (1 << c)]
        dst = torch.full((len(comps) * n + 8,), 5.0, device="cuda")
        sim.read_fields_ptr(mask, dst[offset:].data_ptr())
        got = dst.cpu().numpy()
        assert np.array_equal(got[offset:offset + len(comps) * n].view(np.int32), host[comps].reshape(-1).view(np.int32))
        assert (got[:offset] == 5.0).all() and (got[offset + len(comps) * n:] == 5.0).all()
    if not kw:
        assert np.array_equal(host.view(np.int32), f.view(np.int32))
    sim.close()


def test_nothing_is_read_after_a_timeout(cuda_device):
    shape = (40, 40, 40)
    sim = fdtd.Sim(shape, np.ones(shape), DT, timeout_s=0.2)
    sim.write_fields(torch.as_tensor(wl.random_fields(shape, 1)).cuda())
    sim.debug_set(fdtd.DEBUG_SKIP_PUBLISH, 3)
    sim.step(30)
    out = torch.full((6,) + shape, 5.0, device="cuda")
    with pytest.raises(fdtd.FdtdError) as e:
        sim.read_fields(out=out)
    assert e.value.status == fdtd.FDTD_ERR_TIMEOUT
    assert (out == 5.0).all()
    sim.debug_set(fdtd.DEBUG_NONE)
    sim.write_fields(torch.zeros((6,) + shape, device="cuda"))  # clears the error
    assert (sim.read_fields() == 0).all()
    sim.close()
