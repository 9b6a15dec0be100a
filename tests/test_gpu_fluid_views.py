"""The fluid step on fields that start anywhere in a larger buffer: a view whose
first value lies on 8 bytes (4 for FP32) gives the aligned field's results."""
import numpy as np
import pytest
import torch

from paper_2408_14140_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("off_u,off_p", [(1, 0), (0, 1), (1, 1), (3, 2)])
def test_views_off_16_bytes(prec, off_u, off_p):
    from paper_2408_14140_gb300 import api
    from paper_2408_14140_gb300 import build
    build.build()
    n = (32, 16, 64)
    h = 1.0 / 64
    rng = synth.SplitMix64(5)
    u = synth.fourier_field(n, 4, rng, h)
    p = 0.3 * synth.fourier_field(n, 3, rng, h)[0]
    dt = api.field_dtype(prec)

    def view(a, off):
        buf = torch.zeros(a.size + 4, device="cuda", dtype=dt)
        v = buf[off:off + a.size].view(a.shape)
        v.copy_(torch.tensor(np.ascontiguousarray(a), device="cuda"))
        return v

    ctx = api.Context()
    out = []
    for ou, op in ((0, 0), (off_u, off_p)):
        uu, pp = view(u, ou), view(p, op)
        assert uu.data_ptr() % 16 == (ou * uu.element_size()) % 16
        us = ctx.fluid_predictor(uu, pp, h, 1.0, 0.01, (0.1, 0.0, -0.2), 0.1 * h, u_star=view(0 * u, op))
        ctx.level_projection(uu, pp, h, 1.0, 0.1 * h)
        out.append((us.clone(), uu.clone(), pp.clone()))
    ctx.status()
    ctx.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
