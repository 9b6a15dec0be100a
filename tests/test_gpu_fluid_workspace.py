"""The fluid step's documented workspace: two complex grid fields serve the
predictor and one serves the projection, whatever the grid's shape."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [(16, 16, 16), (16, 64, 32), (32, 16, 16), (256, 16, 32), (16, 16, 512)])
def test_documented_workspace_serves(n, prec):
    from paper_2408_14140_gb300 import api
    from paper_2408_14140_gb300 import build
    build.build()
    dt = api.field_dtype(prec)
    gen = torch.Generator(device="cuda").manual_seed(1)
    u = torch.randn((3, n[2], n[1], n[0]), device="cuda", dtype=torch.float64, generator=gen).to(dt)
    p = torch.randn((n[2], n[1], n[0]), device="cuda", dtype=torch.float64, generator=gen).to(dt)
    field = n[0] * n[1] * n[2] * 2 * u.element_size()
    grid = api.make_grid(n, 0.1, prec=prec)
    g = (ctypes.c_double * 3)(0.0, 0.0, 0.0)
    out = []
    for tight in (False, True):
        uu, pp, us = u.clone(), p.clone(), torch.empty_like(u)
        ctx = api.Context(2 * field if tight else 0)
        assert ctx.lib.fluid_predictor(ctx.handle, ctypes.byref(grid), u.data_ptr(), p.data_ptr(), 1.0, 0.01, g, 1e-3,
                                       us.data_ptr(), 0) == api.IB_OK
        torch.cuda.synchronize()
        ctx.close()
        ctx = api.Context(field if tight else 0)
        assert ctx.lib.level_projection(ctx.handle, ctypes.byref(grid), uu.data_ptr(), pp.data_ptr(), 1.0, 1e-3,
                                        0) == api.IB_OK
        torch.cuda.synchronize()
        ctx.status()
        ctx.close()
        out.append((us, uu, pp))
    for a, b in zip(*out):
        assert torch.equal(a, b)
