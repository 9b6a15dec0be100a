"""The FP64 predictor holds every velocity component to the gate relative to that
component's own size, however much larger the others are."""
import numpy as np
import pytest
import torch

from oracle import fluid
from paper_2408_14140_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(64, 32, 16), (16, 32, 32)])
@pytest.mark.parametrize("sizes", [(1.0, 0.7, 1e-4), (1.0, 1e-8, 0.5), (1e-12, 1.0, 1e-6), (3.0, 1e-30, 1e-60),
                                   (1.0, 0.0, 1e-10), (1e-9, 1e-9, 1e-9)])
def test_small_components(n, sizes):
    from paper_2408_14140_gb300 import api
    from paper_2408_14140_gb300 import build
    build.build()
    h = 1.0 / max(n)
    u = synth.fourier_field(n, 5, synth.SplitMix64(8), h) * np.array(sizes)[:, None, None, None]
    p = np.zeros(u.shape[1:])
    dt = 0.2 * h / np.abs(u).max()
    ctx = api.Context()
    us = ctx.fluid_predictor(torch.tensor(u, device="cuda"), torch.tensor(p, device="cuda"), h, 1.1, 0.01 * h * h / dt,
                             (0.0, 0.0, 0.0), dt).cpu().numpy()
    ctx.status()
    ctx.close()
    ref = fluid.predictor(u, p, 1.1, 0.01 * h * h / dt, (0.0, 0.0, 0.0), dt, h)
    for c in range(3):
        assert np.max(np.abs(us[c] - ref[c])) <= 1e-12 * np.max(np.abs(ref[c])), c
