"""Ellipsoid PVF volume integrals and the drag diagnostic on the GPU.

Against the FP64 oracle (1e-12 FP64 fields, 2e-5 FP32 fields, normwise), the
paper's ellipsoid PVF table (Sec. 4.1), the sphere entry point for equal
semi-axes, and boxes too wide for the shared-memory node planes.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2408_14140_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 2e-5}


@pytest.fixture(scope="module")
def api():
    from paper_2408_14140_gb300 import api as a
    from paper_2408_14140_gb300 import build
    build.build()
    return a


def nerr(g, o):
    g = g.detach().double().cpu().numpy()
    o = np.asarray(o)
    return float(np.max(np.abs(g - o)) / max(np.max(np.abs(o)), 1e-300))


def t64(a):
    return torch.tensor(np.asarray(a, dtype=np.float64), device="cuda")


@pytest.mark.parametrize("prec", [0, 1])
def test_ellipsoid_integrals_match_oracle(api, prec):
    N = 48
    h = 1.0 / N
    rng = synth.SplitMix64(17)
    u = synth.fourier_field((N,) * 3, 6, rng, h)
    if prec == 1:
        u = u.astype(np.float32).astype(np.float64)
    P = 6
    X = rng.uniforms(3 * P).reshape(P, 3)  # anywhere, seams included
    ax = (3.0 + 6.0 * rng.uniforms(3 * P).reshape(P, 3)) * h
    ctx = api.Context()
    ug = torch.tensor(u, device="cuda", dtype=api.field_dtype(prec))
    Iu, Irxu, vol = ctx.particle_volume_integrals_ellipsoid(ug, h, t64(X), t64(ax))
    ctx.status()
    o = oracle.volume_integrals_ellipsoid((N,) * 3, h, (0, 0, 0), u, X, ax)
    assert nerr(Iu, o[0]) <= TOL[prec]
    assert nerr(Irxu, o[1]) <= TOL[prec]
    assert nerr(vol, o[2]) <= 1e-12
    ctx.close()


@pytest.mark.parametrize("doh,val", [(16, 0.4004903567), (32, 0.4016884973)])
def test_ellipsoid_volume_table(api, doh, val):
    """The paper's ellipsoid PVF table (Sec. 4.1): axes (0.4, 0.6, 0.4),
    centre (1, 1, 1), domain 2^3, h = 0.8 / (D/h); printed digits."""
    h = 0.8 / doh
    n = int(round(2.0 / h))
    ctx = api.Context()
    u = torch.zeros((3, n, n, n), device="cuda", dtype=torch.float64)
    _, _, vol = ctx.particle_volume_integrals_ellipsoid(u, h, t64([[1, 1, 1]]), t64([[0.4, 0.6, 0.4]]))
    ctx.status()
    assert abs(float(vol[0]) - val) <= 0.5e-10
    ctx.close()


def test_equal_axes_match_sphere_entry_point(api):
    N = 40
    h = 1.0 / N
    rng = synth.SplitMix64(3)
    u = torch.tensor(synth.fourier_field((N,) * 3, 5, rng, h), device="cuda")
    X = t64([[0.31, 0.62, 0.5], [0.9, 0.05, 0.77]])
    R = t64([0.15, 0.2])
    ctx = api.Context()
    z3 = torch.zeros((2, 3), device="cuda", dtype=torch.float64)
    parts = dict(Xr=X, Ur=z3, Wr=z3, radius=R, rho_p=torch.ones(2, device="cuda", dtype=torch.float64),
                 moff=torch.zeros(3, device="cuda", dtype=torch.int32))
    a = ctx.particle_volume_integrals(u, h, parts)
    b = ctx.particle_volume_integrals_ellipsoid(u, h, X, R[:, None].repeat(1, 3).contiguous())
    ctx.status()
    for x, y in zip(a, b):
        assert nerr(x, y.cpu().numpy()) <= 1e-12
    ctx.close()


def test_wide_box_direct_corners(api):
    """An ellipsoid whose box exceeds the node-plane capacity (70 cells)."""
    N = 96
    h = 1.0 / N
    rng = synth.SplitMix64(8)
    u = synth.fourier_field((N,) * 3, 4, rng, h)
    X = [[0.5, 0.47, 0.52]]
    ax = [[34.5 * h, 12 * h, 20 * h]]
    ctx = api.Context()
    out = ctx.particle_volume_integrals_ellipsoid(torch.tensor(u, device="cuda"), h, t64(X), t64(ax))
    ctx.status()
    o = oracle.volume_integrals_ellipsoid((N,) * 3, h, (0, 0, 0), u, X, ax)
    for g, ref in zip(out, o):
        assert nerr(g, ref) <= 1e-12
    ctx.close()


def test_drag_force_matches_oracle(api):
    rng = np.random.default_rng(4)
    Fib, Inew, Iold = (rng.normal(size=(9, 3)) for _ in range(3))
    ctx = api.Context()
    FD = ctx.particle_drag_force(t64(Fib), t64(Inew), t64(Iold), 1.3, 2e-3)
    ctx.status()
    ref = oracle.drag_force(Fib, Inew, Iold, 1.3, 2e-3)
    assert nerr(FD, ref) <= 1e-15
    ctx.close()


# boxes of 40/41 cells (one and a half warps of a row), of 64 cells (the widest
# with node planes) and 65, tall and flat ones, an ellipsoid below a cell, and
# a whole box per CTA or a plane or two per CTA
@pytest.mark.parametrize("split", [0, 1, 32])
def test_cell_classes_and_box_sizes(api, split):
    N = 80
    h = 1.0 / N
    rng = synth.SplitMix64(21)
    u = synth.fourier_field((N,) * 3, 4, rng, h)
    half = np.array([[18.5, 18.9, 2.2], [31.0, 3.0, 31.9], [2.0, 30.6, 31.4], [1.5, 2.5, 37.0],
                     [0.2, 0.4, 0.3], [4.0, 4.0, 4.0]])
    X = np.array([[40, 40, 40], [40.5, 40.25, 12], [0.3, 40, 79.9], [20, 60.1, 40], [33.2, 41.9, 7.5], [16, 16, 16]])
    ctx = api.Context()
    ctx.set_volume_split(split)
    out = ctx.particle_volume_integrals_ellipsoid(torch.tensor(u, device="cuda"), h, t64(X * h), t64(half * h))
    ctx.status()
    ref = oracle.volume_integrals_ellipsoid((N,) * 3, h, (0, 0, 0), u, X * h, half * h)
    for g, r in zip(out, ref):
        assert nerr(g, r) <= TOL[0]
    # cells outside take no part, whatever they hold
    v = torch.full((3, N, N, N), float("nan"), device="cuda", dtype=torch.float64)
    v[:, 8:24, 8:24, 8:24] = torch.tensor(u[:, 8:24, 8:24, 8:24], device="cuda")
    part = ctx.particle_volume_integrals_ellipsoid(v, h, t64(X[5:] * h), t64(half[5:] * h))
    for g, r in zip(part, out):
        assert torch.equal(g[0], r[5])
    ctx.close()


# spheres: boxes of 40 cells (the widest tabulated) and 41 to 43, a box of more
# than a warp's width with seams, one of a few cells, one below a cell
@pytest.mark.parametrize("split", [0, 1, 32])
@pytest.mark.parametrize("prec", [0, 1])
def test_sphere_box_sizes(api, prec, split):
    N = 48
    h = 1.0 / N
    rng = synth.SplitMix64(33)
    u = synth.fourier_field((N,) * 3, 4, rng, h)
    if prec == 1:
        u = u.astype(np.float32).astype(np.float64)
    half = np.array([18.9, 19.6, 16.3, 3.0, 1.6, 0.3])
    X = np.array([[24, 24, 24], [24, 23.5, 24.2], [0.1, 47.8, 30.3], [12, 12, 12], [40.2, 7.7, 9.1], [30.4, 5.6, 20.1]])
    P = len(half)
    z3 = torch.zeros((P, 3), device="cuda", dtype=torch.float64)
    parts = dict(Xr=t64(X * h), Ur=z3, Wr=z3, radius=t64(half * h), rho_p=torch.ones(P, device="cuda", dtype=torch.float64),
                 moff=torch.zeros(P + 1, device="cuda", dtype=torch.int32))
    ctx = api.Context()
    ctx.set_volume_split(split)
    out = ctx.particle_volume_integrals(torch.tensor(u, device="cuda", dtype=api.field_dtype(prec)), h, parts)
    ctx.status()
    ref = oracle.volume_integrals((N,) * 3, h, (0, 0, 0), u, X * h, half * h)
    for g, r in zip(out, ref):
        assert nerr(g, r) <= 1e-12
    ctx.close()
