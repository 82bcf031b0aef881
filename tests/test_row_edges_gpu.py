"""Systolic kernel where rows of its tiles lie outside the domain in y: their
warps skip the half-steps.  Extents around the tile's 15 rows and the 16 y
slots, whole lives of tiles in one launch (more steps than a tile's extent),
launches that end inside one, and sources on the edge rows; bit for bit
against the naive schedule."""
import pytest
import torch

from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DT = wl.DT_DEFAULT


def run(shape, calls, scheme, **kw):
    nz, ny, nx = shape
    sim = fdtd.Sim(shape, wl.random_eps(shape, 5), DT, scheme=scheme, max_source_steps=64, **kw)
    sim.write_fields(torch.as_tensor(wl.random_fields(shape, 5, zero_pec_walls=False)).cuda())
    sim.add_source(2, nx // 2, ny - 1, nz // 2, wl.sine_source(50, DT))
    sim.add_source(1, nx // 3, 0, nz - 1, wl.sine_source(20, DT, 5.0))
    for n in calls:
        sim.step(n)
    out = sim.read_fields().view(torch.int32)
    sim.close()
    return out


@pytest.mark.parametrize("ny", [1, 2, 14, 15, 16, 17, 29, 30, 31, 47])
@pytest.mark.parametrize("tile,kw", [
    ("31x15x12", {}), ("31x15x8", {}), ("31x15x12", {"storage": "f16"}),
    ("31x15x12", {"boundary": "graded", "absorber": (1, 0.5, 3), "storage": "bf16"})])
def test_rows_outside_the_domain(cuda_device, ny, tile, kw):
    shape = (27, ny, 40)
    want = run(shape, [60], "naive", **kw)
    assert torch.equal(run(shape, [60], "systolic", tile=tile, **kw), want)
    assert torch.equal(run(shape, [7, 40, 13], "systolic", tile=tile, **kw), want)
