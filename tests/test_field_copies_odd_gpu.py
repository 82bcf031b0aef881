"""fdtd_write_fields and fdtd_read_fields on device addresses that no float may have:
copied byte by byte, as they were before a kernel took the aligned ones; and rows of
a few values, which take fewer threads than a quarter warp.
"""
import numpy as np
import pytest
import torch

from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [{}, {"storage": "f16"}, {"storage": "bf16"}])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_addresses_between_floats(cuda_device, kw, offset):
    shape = (4, 7, 36)
    f = wl.random_fields(shape, 7, zero_pec_walls=False)
    sim = fdtd.Sim(shape, 2.0, wl.DT_DEFAULT, **kw)
    sim.write_fields(f)
    host = np.empty((6,) + shape, np.float32)
    sim.read_fields_ptr(0x3F, host.ctypes.data)
    src = torch.zeros(f.nbytes + 16, dtype=torch.uint8, device="cuda")
    src[offset:offset + f.nbytes] = torch.from_numpy(f.reshape(-1).view(np.uint8).copy()).cuda()
    sim.write_fields(np.zeros_like(f))
    sim.write_fields_ptr(src.data_ptr() + offset)
    dst = torch.full((2 * f.nbytes // 6 + 16,), 7, dtype=torch.uint8, device="cuda")
    sim.read_fields_ptr(0x12, dst.data_ptr() + offset)
    sim.close()
    got = dst.cpu().numpy()
    assert np.array_equal(got[offset:offset + 2 * f.nbytes // 6], host[[1, 4]].reshape(-1).view(np.uint8))
    assert (got[:offset] == 7).all() and (got[offset + 2 * f.nbytes // 6:] == 7).all()


@pytest.mark.parametrize("kw", [{}, {"storage": "f16"}])
@pytest.mark.parametrize("nx", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("rows", [(1, 1), (300, 7), (2, 2500)])
def test_narrow_rows(cuda_device, kw, nx, rows):
    shape = (*rows, nx)
    f = wl.random_fields(shape, 9, zero_pec_walls=False)
    sim = fdtd.Sim(shape, 2.0, wl.DT_DEFAULT, **kw)
    sim.write_fields(torch.from_numpy(f).cuda())
    got = sim.read_fields().cpu().numpy()
    one = sim.read_fields(mask=0x20).cpu().numpy()
    sim.close()
    ref = f.astype(np.float16).astype(np.float32) if kw else f
    assert np.array_equal(got, ref) and np.array_equal(one[0], ref[5])


# few rows, whose parts go over blocks (in groups of four values and not), and rows
# enough that a thread takes four, the last of them short of four
@pytest.mark.parametrize("kw", [{}, {"storage": "f16"}])
@pytest.mark.parametrize("shape", [(1, 1, 20001), (1, 1, 20000), (3, 3, 1030), (2, 3, 1028), (300, 131, 30), (301, 131, 29),
                                   (250, 160, 17)])
def test_few_long_rows_and_many_short_ones(cuda_device, kw, shape):
    f = wl.random_fields(shape, 11, zero_pec_walls=False)
    sim = fdtd.Sim(shape, 2.0, wl.DT_DEFAULT, scheme="naive", **kw)
    ref = f.astype(np.float16).astype(np.float32) if kw else f
    sim.write_fields(torch.from_numpy(f).cuda())
    got = sim.read_fields().cpu().numpy()
    assert np.array_equal(got, ref)
    sim.write_fields(np.zeros_like(f))
    sim.write_fields(f)  # from the host: a component at a time
    host = np.empty((2,) + shape, np.float32)
    sim.read_fields_ptr(0x28, host.ctypes.data)
    sim.close()
    assert np.array_equal(host, ref[[3, 5]])
