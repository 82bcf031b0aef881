"""A call of no steps launches nothing, whatever the schedule."""
import pytest
import torch

from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [{"scheme": "naive"}, {}, {"tile": "31x15x12"}, {"tile": "31x15x15"}, {"cluster": (2, 1, 1)}])
@pytest.mark.parametrize("shape", [(5, 6, 7), (20, 21, 40)])
def test_no_launch(cuda_device, kw, shape):
    f = torch.as_tensor(wl.random_fields(shape, 1)).cuda()
    sim = fdtd.Sim(shape, 2.0, wl.DT_DEFAULT, **kw)
    sim.write_fields(f)
    sim.step(0)
    assert sim.launch_count == 0 and sim.current_step == 0
    assert torch.equal(sim.read_fields(), f)
    sim.close()
