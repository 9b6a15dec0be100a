"""The fluid step's transforms at every line length and on extreme values.

Each axis length has kernels of its own (radix schedules, lines per CTA, lanes
per row), for FP32 and for FP64 fields (64-bit block fixed point), so every
length is run along every axis against the FP64 oracle, at the library's gates
(normwise, 1e-12 and 2e-5).  The pressure is compared where the solve's
amplification of its smallest modes, at most (n_a n_b / pi^2)^2 of the two
longest axes over the lowest mode's (n / 2 pi)^2, keeps 2^-53 (2^-24) inside
the gate: FP64 with axes of at most 128."""
import numpy as np
import pytest
import torch

from oracle import fluid
from paper_2408_14140_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 2e-5}
SIZES = [(16, 16, 16), (1024, 16, 16), (16, 1024, 16), (16, 16, 1024), (512, 32, 16), (16, 512, 32), (32, 16, 512),
         (256, 16, 128), (128, 256, 16), (16, 128, 256), (64, 32, 64), (32, 64, 32)]


@pytest.fixture(scope="module")
def api():
    from paper_2408_14140_gb300 import api as a
    from paper_2408_14140_gb300 import build
    build.build()
    return a


def nerr(g, o):
    g = g.detach().double().cpu().numpy()
    return float(np.max(np.abs(g - o)) / np.max(np.abs(o)))


def inputs(n, prec, seed):
    rng = synth.SplitMix64(seed)
    h = 1.0 / max(n)
    u = synth.fourier_field(n, 6, rng, h)
    p = 0.3 * synth.fourier_field(n, 4, rng, h)[0]
    u += 0.01 * np.random.RandomState(seed).standard_normal(u.shape)  # every mode present
    if prec == 1:
        u, p = u.astype(np.float32).astype(np.float64), p.astype(np.float32).astype(np.float64)
    return h, u, p


def dev(a, dtype):
    return torch.tensor(a, device="cuda", dtype=dtype)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", SIZES)
def test_every_line_length(api, n, prec):
    h, u, p = inputs(n, prec, 11)
    rho, dt, dtype = 1.1, 0.05 * h, api.field_dtype(prec)
    ctx = api.Context()
    for mu in (0.0, 0.5 * h):
        us = ctx.fluid_predictor(dev(u, dtype), dev(p, dtype), h, rho, mu, (0.1, 0.0, -1.0), dt)
        assert nerr(us, fluid.predictor(u, p, rho, mu, (0.1, 0.0, -1.0), dt, h)) <= TOL[prec]
    u_ref, p_ref = fluid.projection(u, p, rho, dt, h)
    ug, pg = dev(u, dtype), dev(p, dtype)
    ctx.level_projection(ug, pg, h, rho, dt)
    ctx.status()
    assert nerr(ug, u_ref) <= TOL[prec]
    if prec == 0 and max(n) <= 128:
        assert nerr(pg, p_ref) <= TOL[prec]
    ctx.close()


@pytest.mark.parametrize("k", [-900, 700])
def test_projection_scales_by_powers_of_two(api, k):
    """The projection is linear, and its fixed-point blocks are scaled by powers
    of two, so a scaled input gives the scaled result bit for bit."""
    n = (32, 64, 16)
    h, u, p = inputs(n, 0, 12)
    ctx = api.Context()
    out = []
    for s in (1.0, 2.0 ** k):
        ug, pg = dev(u * s, torch.float64), dev(p * s, torch.float64)
        ctx.level_projection(ug, pg, h, 1.0, 1e-3)
        out.append((ug / s, pg / s))
    ctx.status()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    ctx.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_zero_and_nonfinite_fields(api, prec):
    """A field at rest stays at rest exactly; a NaN or an infinity in one cell
    leaves no finite value of the solve behind."""
    n, dtype = (32, 16, 64), api.field_dtype(prec)
    ctx = api.Context()
    z = torch.zeros((3, n[2], n[1], n[0]), device="cuda", dtype=dtype)
    p = torch.zeros((n[2], n[1], n[0]), device="cuda", dtype=dtype)
    assert not ctx.fluid_predictor(z, p, 0.1, 1.0, 0.01, (0.0, 0.0, 0.0), 1e-2).any()
    ctx.level_projection(z, p, 0.1, 1.0, 1e-2)
    assert not z.any() and not p.any()
    for bad in (float("nan"), float("inf")):
        u = torch.ones_like(z)
        u[1, 5, 3, 7] = bad
        assert not torch.isfinite(ctx.fluid_predictor(u, p, 0.1, 1.0, 0.01, (0.0, 0.0, 0.0), 1e-2)[1]).any()
        ctx.level_projection(u, p.clone(), 0.1, 1.0, 1e-2)
        assert not torch.isfinite(u).any()
    ctx.status()
    ctx.close()


@pytest.mark.parametrize("n", [(16, 32, 64), (64, 16, 16)])
@pytest.mark.parametrize("scale,cfl", [(1.0, 5.0), (2.0 ** 500, 0.1), (2.0 ** -500, 0.1), (1.0, 0.1)])
def test_predictor_beyond_the_fixed_point_range(api, n, scale, cfl):
    """FP64 right-hand sides outside the fixed-point kernel's range (Courant
    number above 2, |u| beyond 2^400) and inside it, and a pressure of zero:
    all at the FP64 gate.  Scaling u by s, p by s^2 and dt by 1/s scales the
    step by s."""
    h, u, p = inputs(n, 0, 13)
    dt = cfl * h / np.abs(u).max()
    ctx = api.Context()
    for q in (p, 0 * p):
        ref = fluid.predictor(u, q, 1.0, 0.01, (0.0, 0.0, 0.0), dt, h)
        us = ctx.fluid_predictor(dev(u * scale, torch.float64), dev(q * scale * scale, torch.float64), h, 1.0,
                                 0.01 * scale, (0.0, 0.0, 0.0), dt / scale)
        assert nerr(us / scale, ref) <= TOL[0]
    ctx.status()
    ctx.close()
