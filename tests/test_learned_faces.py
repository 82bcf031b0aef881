"""The learned layer's kernels over the faces' patches: every shape a face can
have, on the GPU against the FP64 learned-boundary step; and the layer's tanh,
emulated in float32 on the CPU, against float64.
"""
import numpy as np
import pytest
import torch

from helpers import rel_l2_per_field
from oracle import mlp
from paper_2502_20610_gb300 import fdtd
from paper_2502_20610_gb300 import workloads as wl

DT = wl.DT_DEFAULT


# one cell, one-cell and two-cell thick domains (one face, no second plane),
# faces smaller than, equal to and one over a 16 x 4 patch, a CTA's run over
# several faces, more patches than CTAs
@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 5, 9), (7, 1, 20), (6, 17, 1), (2, 2, 2), (3, 3, 3), (4, 16, 16),
                                   (5, 17, 18), (9, 6, 33), (40, 70, 50)])
def test_learned_step_over_face_shapes(cuda_device, shape):
    eps = wl.random_eps(shape, 10)
    f0 = wl.random_fields(shape, 10)
    p = mlp.unpack(mlp.init_params(11))
    p["W3"] *= 0.05  # a tame random network
    th32 = mlp.pack(p).astype(np.float32)
    sim = fdtd.Sim(shape, eps, DT, scheme="naive", boundary="learned", learned=(4, th32))
    sim.write_fields(torch.as_tensor(np.asarray(f0, np.float32)).cuda())
    sim.step(3)
    sim.step(1)
    got = sim.read_fields().cpu().numpy()
    sim.close()
    ref, _ = mlp.learned_run(shape, eps, np.asarray(f0, np.float32).astype(np.float64), 4, th32.astype(np.float64),
                             thickness=4, dt=DT)
    # the bound of the learned-step test: FP32 states over a few steps
    assert max(rel_l2_per_field(got, ref).values()) < 1e-4


def test_tanh_form():
    """tanh_fast of csrc/mlp.cu, operation by operation (its exponential and
    reciprocal rounded to nearest): two units in the last place at most."""
    f = np.float32

    def fma(a, b, c):
        return (np.asarray(a, np.float64) * np.asarray(b, np.float64) + np.asarray(c, np.float64)).astype(f)

    x = np.concatenate([np.linspace(1e-6, 12, 1000001), np.logspace(-30, 1, 300001)]).astype(f)
    a = np.where(x > 10, f(10), x)
    t = (a * a).astype(f)
    e = np.exp2((a * f(2.885390081777927)).astype(f)).astype(f)
    small = a < 1
    n = np.where(small, ((a * t).astype(f) * fma(t, fma(t, f(27), f(2772)), f(45045))).astype(f), f(2))
    d = np.where(small, fma(t, fma(t, fma(t, f(28), f(3150)), f(62370)), f(135135)), (e + f(1)).astype(f))
    y = fma(-n, (1 / d.astype(np.float64)).astype(f), np.where(small, a, f(1)))
    ref = np.tanh(x.astype(np.float64))
    assert (np.abs(y - ref) / np.spacing(ref.astype(f))).max() < 2.0
