"""CPU model of the register kernel's face buffers with whole columns
(csrc/systolic_reg.cu).

The model of test_schedule.py with what the kernel does since columns are
stored whole: a tile's top y and x faces carry every row of the tile, rows
outside the grid in z included, a step's shells are read with those rows, and
the buffers' period is a tile's rows longer than the grid.  Every row of a read
column must be the level and the cell it should be.
"""
import inspect

import numpy as np
import pytest

import test_schedule as ts

TILES = [(31, 15, 12), (31, 15, 8)]

CHANGES = (
    # step shells: rows outside the grid in z are read too (a tile's first
    # load takes the rows inside only)
    ("        m = indom(x, y, z)\n        x, y, z = x[m], y[m], z[m]\n        zpl = z == b[2] - 1\n",
     "        m = indom(x, y, np.clip(z, 0, nz - 1)) & (indom(x, y, z) | ((tag == 'step') & (z > b[2] - 1)))\n"
     "        x, y, z = x[m], y[m], z[m]\n        zpl = z == b[2] - 1\n"),
    # faces: whole columns
    ("        for sel, buf, (i0, i1) in (((y == b[1] + n[1] - 1), Y, (y, x)), ((x == b[0] + n[0] - 1), X, (x, y))):\n",
     "        x, y, z = box(b, tuple(b[a] + n[a] for a in range(3)))\n"
     "        m = indom(x, y, np.clip(z, 0, nz - 1))\n        x, y, z = x[m], y[m], z[m]\n"
     "        for sel, buf, (i0, i1) in (((y == b[1] + n[1] - 1), Y, (y, x)), ((x == b[0] + n[0] - 1), X, (x, y))):\n"),
)


def whole_column_model():
    src = inspect.getsource(ts.run_face_model)
    for a, b in CHANGES:
        assert src.count(a) == 1, a
        src = src.replace(a, b)
    scope = dict(vars(ts))
    exec(src, scope)
    return scope["run_face_model"]


def period(nz, tz):
    """The kernel's period: room for the grid's rows and a tile's less one, in whole z-blocks."""
    return ts.face_period(nz + tz - 1, tz)


@pytest.mark.parametrize("N,T", [((45, 33, 20), 25), ((20, 17, 9), 40), ((1, 1, 1), 5), ((20, 33, 24), 30), ((9, 20, 25), 30), ((9, 20, 12), 30)])
@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("n", TILES)
def test_levels_and_coverage(N, T, order, n):
    errors, count, F = whole_column_model()(N, T, period(N[2], n[2]), n_cta=5, seed=3 + order, order=order, n=n)
    assert not errors, errors[:5]
    assert np.all(count == 1)
    assert np.all(F == T - 1)


def test_a_period_of_the_grid_alone_is_caught():
    bad = 0
    for seed in range(6):
        errors, _, _ = whole_column_model()((40, 20, 36), 50, 36, n_cta=5, seed=seed, n=(31, 15, 12))
        bad += bool(errors)
    assert bad
