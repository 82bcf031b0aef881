"""The default systolic tile: 8 rows on domains whose tiles all find an SM, 12
elsewhere, in cluster pairs and with conducting cells.  The choice shows in
the workspace's size, which must equal that of the tile asked for by name."""
import ctypes

import pytest

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


@pytest.mark.parametrize("kw", [{"cluster": (2, 1, 1)}, {"boundary": "graded", "absorber": (4, 0.5, 3)},
                                {"steps_per_launch": 5000}])
def test_forms_with_12_rows_only(kw):
    shape = (40, 40, 40)
    assert size(shape, **kw) == size(shape, tile="31x15x12", **kw)
