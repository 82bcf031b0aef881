"""The layer kernel's own tanh, as it runs, against float64.

With first-layer weights of 0 and a third layer that picks one unit, a face cell's
correction is r tanh(b2); one value of 18 in its stencil makes r = sqrt(18^2 / 324) = 1
exactly, and the tangential E of a low face, which the Yee step leaves alone, starts at
0: what is read back is the tanh itself, rounded nowhere else.
"""
import numpy as np
import pytest
import torch

from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
SHAPE = (6, 7, 8)  # nz, ny, nx
# Ey, Ez beside an Ey on the face x = 0, and Ex beside an Ez on the face y = 0
AT = [(1, 2, 3, 0), (2, 2, 3, 0), (0, 3, 0, 4)]


def layer_tanh(ts):
    """tanh of `ts` (6 of them, for the outputs Ex..Hz) as the layer computes it, the three that low faces show."""
    w1, b1 = np.zeros((64, 324)), np.zeros(64)
    w2, b2 = np.zeros((64, 64)), np.zeros(64)
    w3, b3 = np.zeros((6, 64)), np.zeros(6)
    for o in range(6):
        b2[10 * o + 1], w3[o, 10 * o + 1] = ts[o], 1.0
    params = np.concatenate([a.ravel() for a in (w1, b1, w2, b2, w3, b3)]).astype(np.float32)
    f = torch.zeros((6,) + SHAPE, device="cuda")
    f[1, 2, 2, 0] = 18.0
    f[2, 4, 0, 4] = 18.0
    sim = fdtd.Sim(SHAPE, 1.0, wl.DT_DEFAULT, scheme="naive", boundary="learned", learned=(1, params))
    sim.write_fields(f)
    sim.step(1)
    out = sim.read_fields().cpu().numpy()
    sim.close()
    return np.array([out[a] for a in AT], np.float32)


# The bound: tanhf's own, 2 units in the last place.  (All floats from 2^-14 to 12 on the
# GPU: 1.25 at most here, near 1, and 1.82 for tanhf.)
def test_within_two_units(cuda_device):
    rng = np.random.default_rng(1)
    t = np.concatenate([np.linspace(0.9, 1.4, 180), np.logspace(-6, 1.2, 120), rng.uniform(0, 3, 90)]).astype(np.float32)
    t = np.concatenate([t, -t[::7], [np.float32(0.0), np.nextafter(np.float32(1), np.float32(0)), 1, 10, 30, np.inf]]).astype(np.float32)
    t = t[:len(t) // 3 * 3].reshape(-1, 3)
    got = np.stack([layer_tanh([c, a, b, 0, 0, 0]) for a, b, c in t])
    ref = np.tanh(t.astype(np.float64))
    ulp = np.abs(got - ref) / np.spacing(np.maximum(np.abs(ref), 1e-30).astype(np.float32))
    print(f"{t.size} values, {ulp.max():.2f} units in the last place at most")
    assert ulp.max() <= 2.0
    assert (np.sign(got) == np.sign(t)).all() and (np.abs(got) <= 1.0).all()
