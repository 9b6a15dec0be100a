"""Kept plans and plain volume integrals tell the cells of alpha 1 apart by the
same limit: over many radii and places, with cell centres on the limit to the
last bit, no cell is counted twice or left out (one cell is 1e-4 or more of a
sphere of these sizes; the sums agree to rounding)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("h", [1.0 / 64, 0.1, 3.7e-3])
def test_plan_counts_the_plain_call_s_cells(prec, h):
    from paper_2408_14140_gb300 import api
    from paper_2408_14140_gb300 import build
    build.build()
    N, P = 64, 600
    rs = np.random.RandomState(int(1 / h))
    R = rs.uniform(1.0, 12.0, P) * h
    X = rs.uniform(20.0, 44.0, (P, 3)) * h
    # limits on a cell centre's distance: centred on a node, R - 0.8661 h = |(a, b, c) + 1/2| h
    k = P // 2
    X[:k] = rs.randint(20, 44, (k, 3)) * h
    R[:k] = (np.sqrt(((rs.randint(0, 6, (k, 3)) + 0.5) ** 2).sum(1)) + 0.8661) * h
    t = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    z = t(np.zeros((P, 3)))
    parts = dict(Xr=t(X), radius=t(R), Ur=z, Wr=z.clone(), rho_p=t(np.ones(P)),
                 moff=torch.zeros(P + 1, device="cuda", dtype=torch.int32))
    gen = torch.Generator(device="cuda").manual_seed(2)
    u = torch.rand((3, N, N, N), device="cuda", dtype=torch.float64, generator=gen).to(api.field_dtype(prec))
    ctx = api.Context()
    plan = api.PvfPlan(ctx, P, 30 ** 3)
    kept = ctx.particle_volume_integrals_keep(u, h, parts, plan)
    planned = ctx.particle_volume_integrals_plan(u, h, parts, plan)
    ctx.status()
    ctx.close()
    for a, b in zip(planned, kept):
        scale = b.abs().amax(dim=tuple(range(1, b.dim())), keepdim=True) if b.dim() > 1 else b.abs()
        big = kept[2] if b.dim() == 1 else kept[2][:, None]
        assert ((a - b).abs() <= 1e-11 * torch.maximum(scale, big)).all()
