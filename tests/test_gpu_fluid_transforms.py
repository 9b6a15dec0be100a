"""Rounding of the FP64 transforms at every long line: without viscosity and
pressure, and with a time step too short for convection to count (dt u / h of
2^-60), the predictor is a forward and an inverse transform of its field, so
what it changes is their rounding.  It is compared with the change that scipy's
FP64 transforms make to the same field, on flat lines (noise, and a constant
with noise) and on smooth ones."""
import numpy as np
import pytest
import scipy.fft
import torch

pytestmark = pytest.mark.gpu


def fields(n, rs):
    shape = (n[2], n[1], n[0])
    x = sum(np.arange(k).reshape([-1 if a == b else 1 for b in range(3)]) / k for a, k in enumerate(shape))
    return np.stack([rs.standard_normal(shape), 1.0 + 1e-3 * rs.standard_normal(shape),
                     np.cos(2 * np.pi * x) + 0.3 * np.sin(6 * np.pi * x + 1.0)])


@pytest.mark.parametrize("length", [128, 256, 512, 1024])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_no_larger_than_fp64_transforms(length, axis):
    from paper_2408_14140_gb300 import api
    from paper_2408_14140_gb300 import build
    build.build()
    n = [16, 16, 16]
    n[axis] = length
    u = fields(n, np.random.RandomState(length + axis))
    p = torch.zeros((n[2], n[1], n[0]), device="cuda", dtype=torch.float64)
    ctx = api.Context()
    us = ctx.fluid_predictor(torch.tensor(u, device="cuda"), p, 1.0, 1.0, 0.0, (0.0, 0.0, 0.0), 2.0 ** -60).cpu().numpy()
    ctx.status()
    ctx.close()
    for c in range(3):
        ref = scipy.fft.irfftn(scipy.fft.rfftn(u[c]), s=u[c].shape)
        rms = lambda a: np.sqrt(np.mean(a * a))
        assert rms(us[c] - u[c]) <= rms(ref - u[c]), c
