"""Markers many periods away from the grid: first cells near, beyond a period
and beyond 2^30 cells, against the oracle (both precisions and kernels)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2408_14140_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("periods", [0, -1, 1, -3, 1000, -(2 ** 20), 2 ** 28])
@pytest.mark.parametrize("delta", [0, 1])
@pytest.mark.parametrize("prec", [0, 1])
def test_far_markers_wrap(prec, delta, periods):
    from paper_2408_14140_gb300 import api
    from paper_2408_14140_gb300 import build
    build.build()
    N = 16
    h = 1.0 / N  # positions and their quotients by h are exact, so both sides see the same offsets
    rng = synth.SplitMix64(4)
    u = synth.fourier_field((N,) * 3, 3, rng, h)
    if prec:
        u = u.astype(np.float32).astype(np.float64)
    M = 300
    X = np.floor(rng.uniforms(3 * M).reshape(M, 3) * 2 ** 12) / 2 ** 12 + periods
    F = rng.uniforms(3 * M).reshape(M, 3) - 0.5
    dV = np.full(M, h ** 3)
    t = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    ctx = api.Context()
    U = ctx.ib_interpolate(torch.tensor(u, device="cuda", dtype=api.field_dtype(prec)), t(X), h, delta=delta)
    f = torch.zeros((3, N, N, N), device="cuda", dtype=api.field_dtype(prec))
    ctx.ib_spread(f, t(X), t(F), t(dV), h, delta=delta)
    ctx.status()
    tol = 1e-12 if prec == 0 else 2e-5
    Uo = oracle.interpolate((N,) * 3, h, (0, 0, 0), u, X, delta)
    fo = oracle.spread((N,) * 3, h, (0, 0, 0), X, F, dV, delta)
    assert np.max(np.abs(U.cpu().numpy() - Uo)) <= tol * np.max(np.abs(Uo))
    assert np.max(np.abs(f.double().cpu().numpy() - fo)) <= tol * np.max(np.abs(fo))
    ctx.close()
