"""The transforms on lines of subnormal values: what the format holds of them
comes back.  The symbol's 1/N leaves every one of the N modes rounded to half
the format's smallest value q, and the rounding before it reaches no further
(it is multiplied by at most 1), so a result is off by random sums of N such
errors, of standard deviation below q sqrt(N) / 2; 8 of these bound the largest."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2408_14140_gb300 import api as a
    from paper_2408_14140_gb300 import build
    build.build()
    return a


def field(n, bits, q, seed):
    rs = np.random.RandomState(seed)
    return rs.randint(-(2 ** bits), 2 ** bits + 1, (3, n[2], n[1], n[0])).astype(np.float64) * q


@pytest.mark.parametrize("n", [(16, 32, 64), (64, 16, 16), (512, 16, 16)])
@pytest.mark.parametrize("bits", [20, 40, 44, 51])
def test_subnormal_velocity_comes_back(api, n, bits):
    """Without viscosity and pressure, and with convection's products too small
    to be represented, the FP64 predictor returns its field."""
    q = 2.0 ** -1074
    u = field(n, bits, q, 3)
    p = torch.zeros((n[2], n[1], n[0]), device="cuda", dtype=torch.float64)
    ctx = api.Context()
    us = ctx.fluid_predictor(torch.tensor(u, device="cuda"), p, 0.5, 1.0, 0.0, (0.0, 0.0, 0.0), 1e-3).cpu().numpy()
    ctx.status()
    ctx.close()
    assert np.max(np.abs(us - u)) <= 4.0 * math.sqrt(n[0] * n[1] * n[2]) * q


@pytest.mark.parametrize("bits", [16, 22])
def test_subnormal_projection_fp32(api, bits):
    """The FP32 projection of a subnormal velocity (its x passes are in fixed
    point) against the FP64 one of the same values."""
    n, q = (64, 16, 32), 2.0 ** -149
    u = field(n, bits, q, 4)
    ctx = api.Context()
    out = []
    for dt in (torch.float32, torch.float64):
        v = torch.tensor(u, device="cuda").to(dt)
        p = torch.zeros((n[2], n[1], n[0]), device="cuda", dtype=dt)
        ctx.level_projection(v, p, 1.0, 1.0, 0.25)
        out.append((v.double(), p.double()))
    ctx.status()
    ctx.close()
    tol = (4.0 * math.sqrt(n[0] * n[1] * n[2]) + 2e-5 * 2 ** bits) * q
    for a, b in zip(*out):
        assert (a - b).abs().max().item() <= tol
