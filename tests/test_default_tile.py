"""The default systolic tile: 8 rows on domains whose tiles all find an SM, 12
elsewhere and in cluster pairs.  The choice shows in
the workspace's size, which must equal that of the tile asked for by name."""
import ctypes

import pytest
import torch

from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl


def size(shape, **kw):
    grid, coeffs, boundary = fdtd.make_params(shape, wl.DT_DEFAULT, scheme="systolic", **kw)
    n = ctypes.c_size_t(0)
    status = fdtd.load_library().fdtd_workspace_size(ctypes.byref(grid), ctypes.byref(coeffs), ctypes.byref(boundary),
                                                     ctypes.byref(n))
    assert status == 0
    return n.value


@pytest.mark.parametrize("shape,rows", [
    ((64, 64, 64), 8), ((80, 80, 80), 12), ((1, 1, 1), 8), ((256, 256, 256), 12), ((24, 24, 400), 8),
    ((270, 24, 24), 12), ((300, 8, 8), 8), ((24, 400, 24), 12)])
@pytest.mark.parametrize("kw", [{}, {"storage": "f16"}])
def test_rows_of_the_default_tile(shape, rows, kw):
    assert size(shape, **kw) == size(shape, tile="31x15x%d" % rows, **kw)
    assert size(shape, **kw) != size(shape, tile="31x15x%d" % (20 - rows), **kw)


@pytest.mark.parametrize("kw", [{"cluster": (2, 1, 1)}, {"steps_per_launch": 5000}])
def test_forms_with_12_rows_only(kw):
    shape = (40, 40, 40)
    assert size(shape, **kw) == size(shape, tile="31x15x12", **kw)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(7, 15, 31), (8, 16, 32), (9, 31, 63), (33, 47, 40), (64, 64, 64)])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_lossy_8_rows_give_the_bits_of_12(cuda_device, shape, storage):
    def run(**kw):
        sim = fdtd.Sim(shape, wl.random_eps(shape, 7), wl.DT_DEFAULT, storage=storage, boundary="graded",
                       absorber=(2, 0.5, 3), max_source_steps=64, **kw)
        sim.write_fields(torch.as_tensor(wl.random_fields(shape, 7, zero_pec_walls=False)).cuda())
        sim.add_source(2, shape[2] // 2, shape[1] // 2, shape[0] // 2, wl.sine_source(60, wl.DT_DEFAULT))
        for n in (40, 25, 60):
            sim.step(n)
        out = sim.read_fields().view(torch.int32)
        sim.close()
        return out

    default = run()
    assert torch.equal(default, run(tile="31x15x12"))
    assert torch.equal(default, run(scheme="naive"))
