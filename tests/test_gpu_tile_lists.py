"""Tile lists and slices of the wavefront passes at their edges.

Partial tiles, seams, grids of few tiles, crowded tiles (the second list kernel,
lists longer than the sort's last bucket) and particles of one marker: the
persistent kernel of a context's first call, the wavefront kernels of its later
ones and, for FP32 fields, the group kernels agree bitwise.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2408_14140_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2408_14140_gb300 import api as a
    from paper_2408_14140_gb300 import build
    build.build()
    return a


def sphere_markers(rng, n):
    v = rng.uniforms(3 * n).reshape(n, 3) * 2.0 - 1.0
    return v / np.linalg.norm(v, axis=1, keepdims=True)


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("delta", [0, 1])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,P,per,rad", [
    ((12, 13, 20), 1, 60, 2.4),       # two tiles an axis, the last one of 4, 5 cells
    ((40, 28, 33), 6, 90, 4.3),       # partial tiles and seams on every axis
    ((32, 32, 32), 2, 1900, 3.1),     # more than 512 candidates a tile
    ((48, 40, 32), 9, 1, 3.0),        # one marker a particle
])
def test_forms_agree_bitwise(api, n, P, per, rad, prec, delta, order):
    h = 0.1
    rng = synth.SplitMix64(7 + P)
    u0 = torch.tensor(synth.fourier_field(n, 4, rng, h), device="cuda", dtype=api.field_dtype(prec))
    t = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    X = rng.uniforms(3 * P).reshape(P, 3) * np.array(n) * h  # anywhere, overlaps included
    R = np.concatenate([sphere_markers(rng, per) * rad * h for _ in range(P)])
    parts = dict(Xr=t(X), Ur=t(rng.uniforms(3 * P).reshape(P, 3)), Wr=t(rng.uniforms(3 * P).reshape(P, 3)),
                 radius=t(np.full(P, rad * h)), rho_p=t(np.ones(P)),
                 moff=t(np.arange(P + 1, dtype=np.int32) * per))
    marks = dict(R=t(R), dV=t(np.full(P * per, h ** 3)))
    ctx = api.Context()
    out = []
    for k in range(4 if prec else 3):
        if k == 3:
            ctx.set_pass_kernels("groups")
        u = u0.clone()
        F = ctx.ib_multidirect_forcing(u, h, parts, marks, 4, 0.01, delta=delta, order=order)
        ctx.status()
        out.append((u, F))
    for u, F in out[1:]:
        assert torch.equal(u, out[0][0])
        assert torch.equal(F, out[0][1])
    assert not torch.equal(out[0][0], u0)
    # standalone spreading sums in the list kernels themselves
    Xm = np.repeat(X, per, axis=0) + R
    F = rng.uniforms(3 * P * per).reshape(P * per, 3) - 0.5
    f = u0.clone()
    ctx.ib_spread(f, t(Xm), t(F), marks["dV"], h, delta=delta)
    ctx.status()
    ref = oracle.spread(n, h, (0, 0, 0), Xm, F, np.full(P * per, h ** 3), delta, f=u0.double().cpu().numpy())
    assert np.max(np.abs(f.double().cpu().numpy() - ref)) <= (1e-12 if prec == 0 else 2e-5) * np.max(np.abs(ref))
    ctx.close()
