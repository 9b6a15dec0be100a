"""Sequential forcing of a particle many periods from the grid: first cells
within 2^27 cells of the origin, about 2^29 and 2^30 and far beyond, on either
side.  Positions, their quotients by h and the shifts by whole periods are
exact, so every shifted call repeats the unshifted one bit for bit."""
import numpy as np
import pytest
import torch

from paper_2408_14140_gb300 import synth

pytestmark = pytest.mark.gpu

N, H = (24, 32, 40), 1.0 / 16.0


def forcing(api, prec, delta, passes, shift, arm=(0.0, 0.0, 0.0), Wr=(0.5, 0.25, -0.125)):
    rng = synth.SplitMix64(9)
    u = torch.tensor(synth.fourier_field(N, 3, rng, H), device="cuda", dtype=api.field_dtype(prec)).contiguous()
    R, dV = synth.sphere_markers(5.0 * H, H)
    R = np.floor(R * 2 ** 12) / 2 ** 12
    t = lambda a, dt=torch.float64: torch.tensor(np.ascontiguousarray(a), device="cuda", dtype=dt)
    R += np.array(arm)
    X = np.array([[11.25, 17.5, 20.125]]) * H + shift - np.array(arm)
    parts = dict(Xr=t(X), Ur=t([[0.1, -0.2, 0.3]]), Wr=t([Wr]), radius=t([5.0 * H]), rho_p=t([1.5]),
                 moff=t([0, len(dV)], torch.int32))
    ctx = api.Context()
    ctx.set_pass_kernels(passes)
    F = ctx.ib_multidirect_forcing(u, H, parts, dict(R=t(R), dV=t(dV)), 2, 1e-2, delta=delta)
    ctx.status()
    ctx.close()
    return u, F


@pytest.mark.parametrize("prec,delta,passes", [(0, 0, "wavefront"), (0, 1, "wavefront"), (1, 0, "wavefront"),
                                               (1, 1, "groups"), (1, 0, "resident")])
def test_far_particle_repeats_the_near_one(prec, delta, passes):
    from paper_2408_14140_gb300 import api
    from paper_2408_14140_gb300 import build
    build.build()
    u0, F0 = forcing(api, prec, delta, passes, np.zeros(3))
    for cells in (1000, 2 ** 27 - 40, 2 ** 28, 2 ** 29, 2 ** 30 - 3, 2 ** 32, 2 ** 37):
        for sign in ((1, 1, 1), (-1, 1, -1), (1, 0, 0)):
            shift = np.array([s * (cells // n) * n * H for s, n in zip(sign, N)])
            u, F = forcing(api, prec, delta, passes, shift)
            assert torch.equal(u, u0) and torch.equal(F, F0), (cells, sign)


def test_markers_far_from_their_centre_are_refused():
    """Box bounds hold markers within 2^28 cells of their particle's centre; an
    arm longer than that is reported, not given a wrong box."""
    from paper_2408_14140_gb300 import api
    from paper_2408_14140_gb300 import build
    build.build()
    z = np.zeros(3)
    u0, F0 = forcing(api, 0, 0, "wavefront", z, Wr=z)
    u, F = forcing(api, 0, 0, "wavefront", z, [(2 ** 26 // N[0]) * N[0] * H, 0.0, 0.0], z)
    assert torch.equal(u, u0) and torch.equal(F, F0)
    for cells in (2 ** 29, 2 ** 33):
        with pytest.raises(api.IBError) as e:
            forcing(api, 0, 0, "wavefront", z, [0.0, 0.0, -(cells // N[2]) * N[2] * H], z)
        assert e.value.code == api.IB_ERR_UNSUPPORTED
