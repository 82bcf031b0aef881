"""The learned layer passes a NaN on: one in a cell's stencil makes that cell's
corrections NaN, one in a weight those of every cell whose output it enters, whatever
the NaN's bits (the GPU's own arithmetic makes 0x7fffffff).
"""
import numpy as np
import pytest
import torch

from oracle import mlp
from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DT = wl.DT_DEFAULT
SHAPE = (9, 20, 33)  # nz, ny, nx
NANS = [0x7fffffff, 0xffffffff, 0x7fc00000, 0x7f800001]


def corrected():
    """(6, nz, ny, nx): the values the layer corrects (tangential E on low faces, H on high ones)."""
    nz, ny, nx = SHAPE
    m = np.zeros((6,) + SHAPE, bool)
    for axis, comps in ((2, (1, 2)), (1, (0, 2)), (0, (0, 1))):
        for c in comps:
            lo, hi = [slice(None)] * 3, [slice(None)] * 3
            lo[axis], hi[axis] = 0, SHAPE[axis] - 1
            m[c][tuple(lo)] = True
            m[3 + c][tuple(hi)] = True
    return m


def one_step(fields, params=None):
    kw = dict(boundary="learned", learned=(4, params)) if params is not None else {}
    sim = fdtd.Sim(SHAPE, 2.0, DT, scheme="naive", **kw)
    sim.write_fields(fields)
    sim.step(1)
    out = sim.read_fields().cpu().numpy()
    sim.close()
    return out


def float_of(bits):
    return np.array([bits], np.uint32).view(np.float32)[0]


def planted(a, at, bits):
    """A copy of `a` with the NaN's very bits at flat index `at`."""
    a = np.ascontiguousarray(a, np.float32).copy()
    a.reshape(-1).view(np.uint32)[at] = bits
    return a


@pytest.mark.parametrize("bits", NANS)
@pytest.mark.parametrize("cell", [(5, 0, 4), (32, 11, 4), (0, 0, 0), (16, 1, 8), (20, 18, 7)])  # x, y, z
def test_in_a_field(cuda_device, bits, cell):
    x, y, z = cell
    params = mlp.init_params(3).astype(np.float32)
    f = planted(wl.random_fields(SHAPE, 3), np.ravel_multi_index((5, z, y, x), (6,) + SHAPE), bits)
    f = torch.from_numpy(f).cuda()
    near = np.zeros(SHAPE, bool)
    near[max(0, z - 1):z + 2, max(0, y - 1):y + 2, max(0, x - 1):x + 2] = True
    expect = np.isnan(one_step(f)) | (corrected() & near)
    assert (corrected() & near).any()
    assert np.array_equal(np.isnan(one_step(f, params)), expect)


# (offset in the parameters, the components it reaches): the centre tap and one
# beyond each low wall in W1, b1, W2, b2, W3 and b3 of output 2
@pytest.mark.parametrize("bits", NANS)
@pytest.mark.parametrize("at,only", [(7 * 324 + 13, None), (7 * 324 + 27 + 12, None), (7 * 324 + 10, None), (7 * 324 + 4, None),
                                     (20736 + 9, None), (20800 + 64 * 5 + 9, None), (24896 + 5, None),
                                     (24960 + 2 * 64 + 3, 2), (25344 + 2, 2)])
def test_in_a_weight(cuda_device, bits, at, only):
    f = torch.from_numpy(wl.random_fields(SHAPE, 4)).cuda()
    m = corrected()
    if only is not None:
        m[[c for c in range(6) if c != only]] = False
    got = one_step(f, planted(mlp.init_params(3), at, bits))
    assert np.array_equal(np.isnan(got), m)


@pytest.mark.parametrize("bits", [0x7f800000, 0xff800000])
@pytest.mark.parametrize("at", [7 * 324 + 13, 7 * 324 + 10, 20800 + 64 * 5 + 9])
def test_an_infinite_weight(cuda_device, bits, at):
    """Infinite products of either sign, and those with zeros, meet in a sum."""
    f = torch.from_numpy(wl.random_fields(SHAPE, 4)).cuda()
    assert np.array_equal(np.isnan(one_step(f, planted(mlp.init_params(3), at, bits))), corrected())
