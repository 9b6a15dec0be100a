"""The predictor's mean velocity grows by dt g, no more and no less: the other
terms sum to zero over a periodic level.  dt g lies 0.45 units between the
field's last bits, so a sum u + dt g rounds by -0.45 units in every cell.  What
is random in the mean is below 8 roundings of that size over sqrt(N)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [(64, 64, 64), (16, 128, 64)])
def test_mean_velocity_follows_the_body_force(n, prec):
    from paper_2408_14140_gb300 import api
    from paper_2408_14140_gb300 import build
    build.build()
    bit = 2.0 ** (-24 if prec else -53)  # the last bit of values in [0.5, 1)
    h = 1.0 / 64
    dt = 0.05 * h
    rs = np.random.RandomState(7)
    u = np.where(rs.rand(3, n[2], n[1], n[0]) < 0.5, -1.0, 1.0) * rs.uniform(0.55, 0.95, (3, n[2], n[1], n[0]))
    u = torch.tensor(u, device="cuda").to(api.field_dtype(prec))
    p = torch.zeros((n[2], n[1], n[0]), device="cuda", dtype=u.dtype)
    g = [(1000 + 0.45) * bit / dt, 0.0, -(700 + 0.45) * bit / dt]
    ctx = api.Context()
    us = ctx.fluid_predictor(u, p, h, 1.0, 0.001, g, dt)
    ctx.status()
    ctx.close()
    grown = (us.double() - u.double()).cpu().numpy().astype(np.longdouble).mean(axis=(1, 2, 3))
    for c in range(3):
        assert abs(float(grown[c] - np.longdouble(dt * g[c]))) <= 8 * 2 * bit / np.sqrt(n[0] * n[1] * n[2]) + 0.02 * bit, c
