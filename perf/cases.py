"""Timed cases of the library: what a particle-laden-flow program asks of it,
from the single sphere of a small box to dense clusters, batches, the fluid
step around the forcing, and one whole time step.

A case is a dict of plain values; ``kind`` says which entry points it calls:

* ``forcing``   Algorithm 1 on one field (sequential or simultaneous order);
* ``batch``     Algorithm 1 and the volume integrals of many independent cases
                through a prepared table (the serving loop's step);
* ``transfer``  the two transfer operators alone, interpolation and spreading;
* ``integrals`` PVF volume integrals before and after (kept plan) and the
                marker force and torque sums;
* ``ellipsoids`` PVF volume integrals of ellipsoids;
* ``predictor``, ``projection``  the fluid step's two halves;
* ``step``      one whole time step on a periodic level.

Sizes come from the benchmark's workloads (256^3 with 64 spheres of 24 cells,
384^3 with 512 spheres of 16 cells, batches of 32^3 to 128^3 boxes), the paper's
single-sphere box (64^3, 20 cells) and ragged variants of them.
"""
import math

import numpy as np
import torch

from paper_2408_14140_gb300 import api, synth

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # one sphere in a small periodic box: the paper's correctness case, all launches and latency
        dict(name="forcing_small_f64", kind="forcing", n0=64, n1=64, n2=64, P=1, D=20.0, phi=0.1, Ns=2, f64=True,
             four=False, simultaneous=False),
        # the benchmark's cluster in the paper's precision
        dict(name="forcing_cluster_f64", kind="forcing", n0=256, n1=256, n2=256, P=64, D=24.0, phi=0.2, Ns=5, f64=True,
             four=False, simultaneous=False),
        # the dense cluster: many small spheres in contact, single-precision fields
        dict(name="forcing_dense_f32", kind="forcing", n0=384, n1=384, n2=384, P=512, D=16.0, phi=0.3, Ns=3, f64=False,
             four=False, simultaneous=False),
        # the wide kernel and the simultaneous order on a ragged grid with a fractional diameter
        dict(name="forcing_fourpoint_f32", kind="forcing", n0=250, n1=203, n2=231, P=40, D=21.5, phi=0.12, Ns=3,
             f64=False, four=True, simultaneous=True),
        # a server's batch: independent boxes of mixed sizes advanced together
        dict(name="batch_f32", kind="batch", cases=48, P=8, D=24.0, Ns=3, f64=False),
        # interpolation and spreading called alone (a solver with its own forcing loop)
        dict(name="transfer_f64", kind="transfer", n0=256, n1=256, n2=256, P=64, D=24.0, phi=0.2, f64=True, four=False),
        # a step's particle sums around the forcing: integrals before and after, force and torque
        dict(name="integrals_f64", kind="integrals", n0=256, n1=256, n2=256, P=64, D=24.0, phi=0.2, f64=True),
        # ellipsoids of unequal axes
        dict(name="ellipsoids_f32", kind="ellipsoids", n0=256, n1=256, n2=256, P=48, D=24.0, phi=0.1, f64=False),
        # momentum predictor, single precision, the benchmark's grid
        dict(name="predictor_f32", kind="predictor", n0=256, n1=256, n2=256, f64=False, mu=1e-3),
        # level projection in the paper's precision on a channel-shaped level
        dict(name="projection_f64", kind="projection", n0=512, n1=128, n2=128, f64=True),
        # a small level's projection in single precision (on finer grids the solve amplifies the rounding of a few
        # nearly checkerboard modes beyond what two 32-bit pressures can be compared by)
        dict(name="projection_f32", kind="projection", n0=64, n1=64, n2=128, f64=False),
        # one whole time step in the paper's precision: predictor, forcing with its sums, projection, particle update
        dict(name="step_f64", kind="step", n0=128, n1=128, n2=128, P=12, D=20.0, phi=0.08, Ns=3, f64=True, mu=2e-3),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(lo, hi):
        base = size(lo, hi)
        return dict(zip(("n0", "n1", "n2"), (max(lo, min(hi, int(base * rng.uniform(0.75, 1.25)))) for _ in range(3))))

    def spheres(n, most):
        D = round(rng.uniform(8.0, 24.0), 2)
        D = min(D, round(0.35 * min(n.values()), 2))
        room = (0.8 * min(n.values()) / D) ** 3 * 0.1 * 6 / math.pi
        return dict(P=max(1, min(size(1, most), int(room))), D=D, phi=round(rng.uniform(0.05, 0.12), 3))

    def power(cells, longest=9):
        while True:
            e = [rng.randint(4, longest) for _ in range(3)]
            if 15 <= sum(e) <= cells:
                return dict(zip(("n0", "n1", "n2"), (1 << k for k in e)))

    kind = rng.choice(["forcing", "forcing", "forcing", "batch", "transfer", "integrals", "ellipsoids", "predictor",
                       "projection", "step"])
    f64 = rng.random() < 0.5
    if kind == "batch":
        return dict(kind=kind, cases=size(2, 48), P=rng.randint(1, 8), D=round(rng.uniform(10.0, 24.0), 2),
                    Ns=rng.randint(1, 4), f64=f64)
    if kind in ("predictor", "projection"):
        more = dict(mu=round(10.0 ** rng.uniform(-4, -1), 6)) if kind == "predictor" else {}
        n = power(23) if f64 else power(24) if more else power(18, 6)
        return dict(kind=kind, **n, f64=f64, **more)
    if kind == "step":
        n = power(20)
        while min(n.values()) < 32:
            n = power(20)
        return dict(kind=kind, **n, **spheres(n, 16), Ns=rng.randint(1, 4), f64=True, mu=round(10.0 ** rng.uniform(-3, -2), 6))
    n = box(48, 288)
    c = dict(kind=kind, **n, **spheres(n, 96), f64=f64)
    if kind == "forcing":
        c.update(Ns=rng.randint(1, 5), four=rng.random() < 0.3, simultaneous=rng.random() < 0.3)
    if kind == "transfer":
        # the interpolated velocity comes in 64 bits whatever the field's type
        c.update(f64=True, four=rng.random() < 0.3)
    return c


# ---------------------------------------------------------------------------
# inputs (made on the GPU from the seed; particle placement on the host)
# ---------------------------------------------------------------------------
RHO_F, EPS_C, G_COLL = 1.0, 1e-4, 9.81
GRAVITY = (0.0, 0.0, 0.0)  # the particles are carried by the flow
BODY = (0.3, 0.0, -0.2)    # the predictor's body force


def _shape(c):
    return (c["n0"], c["n1"], c["n2"])


def _modes_field(n, rs, K=12, amp=1.0, comps=3, shift=0.5):
    """Sum of K random Fourier modes of integer wavenumbers in [-4, 4], as a
    matrix product of the separated phases, [comps, n2, n1, n0] in 64 bits."""
    k = rs.randint(-4, 5, (K, 3))
    k[np.all(k == 0, axis=1)] = 1
    a = rs.standard_normal((comps, K)) * amp / math.sqrt(K)
    ph = rs.uniform(0, 2 * math.pi, K)

    def phase(ax, extra=0.0):
        x = (torch.arange(n[ax], device=DEV, dtype=F64) + shift) / n[ax]
        return 2 * math.pi * x[:, None] * torch.as_tensor(k[:, ax], device=DEV, dtype=F64) + torch.as_tensor(
            np.zeros(K) + extra, device=DEV, dtype=F64)

    ty, tz, tx = phase(1), phase(2, ph), phase(0)
    t = (tz[:, None, :] + ty[None, :, :]).reshape(-1, K)
    left = torch.cat([torch.cos(t), -torch.sin(t)], 1)
    right = torch.cat([torch.cos(tx), torch.sin(tx)], 1)
    out = torch.empty((comps, n[2] * n[1], n[0]), device=DEV, dtype=F64)
    for c in range(comps):
        w = torch.as_tensor(np.concatenate([a[c], a[c]]), device=DEV, dtype=F64)
        torch.mm(left, (right * w).T.contiguous(), out=out[c])
    return out.view(comps, n[2], n[1], n[0])


def _place(P, D, phi, n, rs):
    """Centres (in cells) of P spheres of diameter D placed at random without
    overlap in a centred box of volume fraction phi (a larger one if they do
    not fit)."""
    side = (P * math.pi / 6 * D ** 3 / phi) ** (1 / 3)
    n = np.asarray(n, float)
    while True:
        s = np.minimum(max(side, 1.05 * D), n - 2)
        lo = 0.5 * (n - s) + 0.5 * D
        span = np.maximum(s - D, 0.0)
        cent = np.empty((0, 3))
        for _ in range(200):
            q = lo + span * rs.uniform(size=(512, 3))
            if len(cent):
                d2 = ((q[:, None, :] - cent[None]) ** 2).sum(-1)
                q = q[(d2 >= D * D).all(1)]
            for c in q:
                if len(cent) < P and (not len(cent) or ((cent - c) ** 2).sum(1).min() >= D * D):
                    cent = np.vstack([cent, c])
            if len(cent) == P:
                return cent
        if (s >= n - 2).all():
            raise RuntimeError("the spheres do not fit the grid")
        side *= 1.1


def _dev(a, dtype=F64):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV).to(dtype).contiguous()


def _particles(cent, diam, h, rs):
    """Device dicts of the spheres (centres in cells) and their surface markers."""
    P = len(cent)
    Rs, dVs, off, made = [], [], [0], {}
    for p in range(P):
        if diam[p] not in made:
            made[diam[p]] = synth.sphere_markers(0.5 * diam[p] * h, h)
        R, dV = made[diam[p]]
        Rs.append(R)
        dVs.append(dV)
        off.append(off[-1] + len(dV))
    parts = dict(Xr=_dev(cent * h), Ur=_dev(0.1 * rs.standard_normal((P, 3))), Wr=_dev(0.1 * rs.standard_normal((P, 3))),
                 radius=_dev(0.5 * np.asarray(diam) * h), rho_p=_dev(np.full(P, 1.5)), moff=_dev(off, torch.int32))
    return parts, dict(R=_dev(np.concatenate(Rs)), dV=_dev(np.concatenate(dVs)))


def _inputs(case, seed):
    rs = np.random.RandomState(seed % (1 << 32))
    kind, real = case["kind"], F64 if case["f64"] else torch.float32
    if kind == "batch":
        fields, hs, pl, ml = [], [], [], []
        mix = np.random.RandomState(case["cases"] * 64 + case["P"])  # the boxes' sizes are the case's, not the seed's
        for _ in range(case["cases"]):
            N = int(mix.choice([32, 48, 64, 96, 128]))
            D = mix.uniform(8.0, min(case["D"], 0.4 * N))
            room = max(1, int((0.8 * N / D) ** 3 * 0.12))
            cent = _place(mix.randint(1, min(case["P"], room) + 1), D, 0.1, (N, N, N), rs)
            parts, marks = _particles(cent, [D] * len(cent), 1.0 / N, rs)
            fields.append(_modes_field((N, N, N), rs, 8).to(real).contiguous())
            hs.append(1.0 / N)
            pl.append(parts)
            ml.append(marks)
        parts, marks, ranges, _ = api.pack_batch(pl, ml)
        return dict(fields=fields, hs=hs, parts=parts, marks=marks, ranges=ranges)
    n = _shape(case)
    h = 1.0 / max(n)
    s = dict(n=n, h=h, dt=0.1 * h if kind in ("step", "predictor", "projection") else 1e-3)
    s["u"] = _modes_field(n, rs).to(real).contiguous()
    if kind in ("predictor", "projection", "step"):
        s["p"] = _modes_field(n, rs, K=8, amp=0.3, comps=1, shift=0.0)[0].to(real).contiguous()
    if "P" not in case:
        return s
    cent = _place(case["P"], case["D"], case["phi"], n, rs)
    if kind == "ellipsoids":
        s["Xr"] = _dev(cent * h)
        s["axes"] = _dev(0.5 * case["D"] * h * rs.uniform(0.6, 1.0, (len(cent), 3)))
        return s
    s["parts"], s["marks"] = _particles(cent, [case["D"]] * len(cent), h, rs)
    M = s["marks"]["dV"].numel()
    if kind == "transfer":
        s["X"] = _marker_positions(s["parts"], s["marks"])
    if kind in ("transfer", "integrals"):
        s["F"] = _dev(rs.standard_normal((M, 3)))
    if kind == "integrals":
        s["u1"] = (s["u"].double() + 0.05 * _modes_field(n, rs)).to(real).contiguous()
    return s


def _marker_positions(parts, marks):
    count = torch.diff(parts["moff"]).long()
    return (torch.repeat_interleave(parts["Xr"], count, dim=0) + marks["R"]).contiguous()


def prepare(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    s["case"], s["ctx"] = case, api.Context()
    if "marks" in s and kind in ("forcing", "batch", "step"):
        s["F"] = torch.zeros((s["marks"]["dV"].numel(), 3), dtype=F64, device=DEV)
    if kind == "batch":
        s["table"] = api.BatchTable(s["ctx"], s["fields"], s["hs"], s["ranges"], s["parts"]["Xr"].shape[0])
    elif kind == "transfer":
        s["U"], s["f"] = torch.zeros_like(s["X"]), torch.zeros_like(s["u"])
    elif kind == "integrals":
        s["plan"] = api.PvfPlan(s["ctx"], case["P"], int(case["D"] + 4) ** 3)
    elif kind in ("predictor", "step"):
        s["u_star"] = torch.zeros_like(s["u"])
    return s


def run(s):
    c, ctx = s["case"], s["ctx"]
    kind = c["kind"]
    if kind == "forcing":
        ctx.ib_multidirect_forcing(s["u"], s["h"], s["parts"], s["marks"], c["Ns"], s["dt"],
                                   delta=api.PESKIN4 if c["four"] else api.ROMA3,
                                   order=api.SIMULTANEOUS if c["simultaneous"] else api.SEQUENTIAL, F_out=s["F"])
        return {"u": s["u"], "F": s["F"]}
    if kind == "batch":
        ctx.ib_batch_table_multidirect_forcing(s["table"], s["parts"], s["marks"], c["Ns"], 1e-3, F_out=s["F"])
        I = ctx.ib_batch_table_volume_integrals(s["table"], s["parts"])
        return {"F": s["F"], "I": I, "u": s["fields"]}
    if kind == "transfer":
        delta = api.PESKIN4 if c["four"] else api.ROMA3
        ctx.ib_interpolate(s["u"], s["X"], s["h"], delta=delta, U=s["U"])
        ctx.ib_spread(s["f"], s["X"], s["F"], s["marks"]["dV"], s["h"], delta=delta)
        return {"U": s["U"], "f": s["f"]}
    if kind == "integrals":
        I0 = ctx.particle_volume_integrals_keep(s["u"], s["h"], s["parts"], s["plan"])
        I1 = ctx.particle_volume_integrals_plan(s["u1"], s["h"], s["parts"], s["plan"])
        FT = ctx.particle_force_torque(s["parts"], s["marks"], s["F"], RHO_F)
        return {"I0": I0, "I1": I1, "FT": FT}
    if kind == "ellipsoids":
        return {"I": ctx.particle_volume_integrals_ellipsoid(s["u"], s["h"], s["Xr"], s["axes"])}
    if kind == "predictor":
        return {"u_star": ctx.fluid_predictor(s["u"], s["p"], s["h"], RHO_F, c["mu"], BODY, s["dt"], u_star=s["u_star"])}
    if kind == "projection":
        ctx.level_projection(s["u"], s["p"], s["h"], RHO_F, s["dt"])
        return {"u": s["u"], "p": s["p"]}
    # the whole step
    h, dt, parts, marks = s["h"], s["dt"], s["parts"], s["marks"]
    us = ctx.fluid_predictor(s["u"], s["p"], h, RHO_F, c["mu"], BODY, dt, u_star=s["u_star"])
    s["u"], s["u_star"] = us, s["u"]
    I0 = ctx.particle_volume_integrals(us, h, parts)
    ctx.ib_multidirect_forcing(us, h, parts, marks, c["Ns"], dt, F_out=s["F"])
    I1 = ctx.particle_volume_integrals(us, h, parts)
    F_ib, T_ib = ctx.particle_force_torque(parts, marks, s["F"], RHO_F)
    ctx.level_projection(us, s["p"], h, RHO_F, dt)
    ctx.particle_collide_update(parts, s["n"], h, (RHO_F, *GRAVITY, G_COLL, EPS_C, h), dt, F_ib, T_ib, I1[0], I0[0],
                                I1[1], I0[1])
    return {"u": us, "p": s["p"], "F": s["F"], "Xr": parts["Xr"], "Ur": parts["Ur"], "Wr": parts["Wr"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind, s = case["kind"], 8 if case["f64"] else 4
    if kind in ("predictor", "projection", "step"):
        N = case["n0"] * case["n1"] * case["n2"]
        fft = 2 * 2.5 * N * math.log2(N)  # one real field there and back
        fluid = {"predictor": (7 * s * N, 3 * fft + 250 * N), "projection": (8 * s * N, fft + 100 * N)}
        if kind != "step":
            return {"bytes": fluid[kind][0], "flops": fluid[kind][1]}
        b, f = (sum(v[k] for v in fluid.values()) for k in range(2))
    else:
        b, f = 0, 0
    if kind == "batch":
        # boxes hold about two thirds of the most spheres, of the mean diameter
        P, D, Ns, W = case["cases"] * max(1.0, 0.5 * case["P"]), 0.5 * (8.0 + case["D"]), case["Ns"], 3
    else:
        P, D, Ns, W = case["P"], case["D"], case.get("Ns", 1), 4 if case.get("four") else 3
    M = P * math.pi * D * D
    band = M * (W + 1)                              # cells under some marker's kernel
    inside = P * math.pi / 6 * (D + math.sqrt(3)) ** 3  # cells that a sphere's integral reads
    taps = 12 * M * W ** 3                          # interpolate and spread three components
    if kind == "forcing":
        return {"bytes": 6 * s * band + 56 * M, "flops": Ns * taps}
    if kind == "batch":
        return {"bytes": 6 * s * band + 56 * M + 3 * s * inside, "flops": Ns * taps + 30 * inside}
    if kind == "transfer":
        return {"bytes": 9 * s * band + 104 * M, "flops": taps}
    if kind == "integrals":
        return {"bytes": 6 * s * inside + 56 * M, "flops": 60 * inside}
    if kind == "ellipsoids":
        return {"bytes": 3 * s * inside * 0.51, "flops": 30 * inside * 0.51}
    return {"bytes": b + 6 * s * band + 80 * M + 6 * s * inside, "flops": f + Ns * taps + 60 * inside}


# ---------------------------------------------------------------------------
# the same results in plain 64-bit torch
# ---------------------------------------------------------------------------
def _phi(r, four):
    r = r.abs()
    if four:
        near = (3 - 2 * r + torch.sqrt((1 + 4 * r - 4 * r * r).clamp_min(0))) / 8
        far = (5 - 2 * r - torch.sqrt((-7 + 12 * r - 4 * r * r).clamp_min(0))) / 8
        return torch.where(r <= 1, near, torch.where(r <= 2, far, torch.zeros_like(r)))
    near = (1 + torch.sqrt((1 - 3 * r * r).clamp_min(0))) / 3
    far = (5 - 3 * r - torch.sqrt((1 - 3 * (1 - r) ** 2).clamp_min(0))) / 6
    return torch.where(r <= 0.5, near, torch.where(r <= 1.5, far, torch.zeros_like(r)))


def _stencil(X, n, h, four):
    """Flat cell index and weight of every tap of markers at X, [M, W^3]."""
    W = 4 if four else 3
    s = X / h - 0.5
    first = (torch.floor(s) - 1 if four else torch.floor(s + 0.5) - 1).long()
    o = torch.arange(W, device=DEV)
    i = first[:, :, None] + o
    w = _phi(s[:, :, None] - i.double(), four)
    i = torch.remainder(i, torch.tensor(n, device=DEV)[None, :, None])
    idx = ((i[:, 2, :, None, None] * n[1] + i[:, 1, None, :, None]) * n[0] + i[:, 0, None, None, :]).reshape(len(X), -1)
    return idx, (w[:, 2, :, None, None] * w[:, 1, None, :, None] * w[:, 0, None, None, :]).reshape(len(X), -1)


def _spread_to(f, idx, wt, A):
    for c in range(3):
        f[c].index_add_(0, idx.reshape(-1), (wt * A[:, c, None]).reshape(-1))


def _forcing(u, n, h, parts, marks, Ns, dt, four, simultaneous):
    """Algorithm 1 in place on u [3, cells]; returns F."""
    X = _marker_positions(parts, marks)
    count = torch.diff(parts["moff"]).long()
    Ud = torch.repeat_interleave(parts["Ur"], count, dim=0) + torch.linalg.cross(
        torch.repeat_interleave(parts["Wr"], count, dim=0), marks["R"])
    F = torch.zeros_like(X)
    off = parts["moff"].tolist()
    for a, b in ([(0, off[-1])] if simultaneous else list(zip(off[:-1], off[1:]))):
        idx, wt = _stencil(X[a:b], n, h, four)
        for _ in range(Ns):
            e = Ud[a:b] - (u[:, idx] * wt).sum(-1).T
            F[a:b] += e / dt
            _spread_to(u, idx, wt, e * (marks["dV"][a:b] / h ** 3)[:, None])
    return F


def _integrals(u, n, h, Xr, axes):
    """PVF integrals of the field u [3, n2, n1, n0] over ellipsoids of semi-axes axes [P, 3]."""
    Iu, Ir, vol = [], [], []
    for p in range(len(Xr)):
        lo = torch.floor((Xr[p] - axes[p]) / h).long() - 1
        hi = torch.ceil((Xr[p] + axes[p]) / h).long() + 1
        i = [torch.arange(int(lo[a]), int(hi[a]) + 1, device=DEV) for a in range(3)]
        nd = [((i[a].double() * h - Xr[p, a]) / axes[p, a]) ** 2 for a in range(3)]
        phi = torch.sqrt(nd[2][:, None, None] + nd[1][None, :, None] + nd[0][None, None, :]) - 1
        neg, tot = torch.zeros((), device=DEV, dtype=F64), torch.zeros((), device=DEV, dtype=F64)
        for dz in (slice(0, -1), slice(1, None)):
            for dy in (slice(0, -1), slice(1, None)):
                for dx in (slice(0, -1), slice(1, None)):
                    neg = neg + (-phi[dz, dy, dx]).clamp_min(0)
                    tot = tot + phi[dz, dy, dx].abs()
        al = torch.where(tot > 0, neg / tot, torch.full_like(tot, 0.5)) * h ** 3
        w = [torch.remainder(i[a][:-1], n[a]) for a in range(3)]
        v = u[:, w[2][:, None, None], w[1][None, :, None], w[0][None, None, :]]
        r = [(i[a][:-1].double() + 0.5) * h - Xr[p, a] for a in range(3)]
        rx, ry, rz = r[0][None, None, :], r[1][None, :, None], r[2][:, None, None]
        av = al * v
        Iu.append(av.sum((1, 2, 3)))
        Ir.append(torch.stack([(ry * av[2] - rz * av[1]).sum(), (rz * av[0] - rx * av[2]).sum(),
                               (rx * av[1] - ry * av[0]).sum()]))
        vol.append(al.sum())
    return torch.stack(Iu), torch.stack(Ir), torch.stack(vol)


def _force_torque(parts, marks, F):
    own = torch.repeat_interleave(torch.arange(len(parts["Xr"]), device=DEV), torch.diff(parts["moff"]).long())
    w = F * marks["dV"][:, None]
    z = torch.zeros_like(parts["Xr"])
    return (-RHO_F * z.index_add(0, own, w), -RHO_F * z.index_add(0, own, torch.linalg.cross(marks["R"], w)))


AX = {0: -1, 1: -2, 2: -3}


def _sh(a, axis, k):
    return torch.roll(a, -k, AX[axis])


def _grad(p, h):
    out = []
    for a in range(3):
        d = _sh(p, a, 1) - p
        for b in range(3):
            if b != a:
                d = d + _sh(d, b, 1)
        out.append(0.25 / h * d)
    return torch.stack(out)


def _div(V, h):
    out = 0
    for a in range(3):
        d = V[a] - _sh(V[a], a, -1)
        for b in range(3):
            if b != a:
                d = d + _sh(d, b, -1)
        out = out + 0.25 / h * d
    return out


def _half_angles(n):
    return [math.pi * torch.fft.fftfreq(n[a], device=DEV, dtype=F64).view([-1 if AX[a] == d else 1 for d in (-3, -2, -1)])
            for a in range(3)]


def _convection(u, h, dt):
    out = torch.zeros_like(u)
    for a in range(3):
        dm, dp = u - _sh(u, a, -1), _sh(u, a, 1) - u
        mag = torch.minimum(2 * torch.minimum(dm.abs(), dp.abs()), 0.5 * (dm + dp).abs())
        sl = torch.where(dm * dp > 0, torch.sign(dm + dp) * mag, torch.zeros_like(mag))
        left = u + (0.5 - dt * u[a] / (2 * h)) * sl
        right = _sh(u - (0.5 + dt * u[a] / (2 * h)) * sl, a, 1)
        lv, rv = left[a], right[a]
        zero = torch.zeros_like(lv)
        un = torch.where((lv > 0) & (lv + rv > 0), lv, torch.where((rv < 0) & (lv + rv < 0), rv, zero))
        flux = un * torch.where(un > 0, left, torch.where(un < 0, right, 0.5 * (left + right)))
        out += (flux - _sh(flux, a, -1)) / h
    return out


def _predictor(u, p, n, h, mu, dt):
    nu = mu / RHO_F
    lap = sum((_sh(u, a, 1) - 2 * u + _sh(u, a, -1)) / (h * h) for a in range(3))
    g = torch.tensor(BODY, device=DEV, dtype=F64)[:, None, None, None]
    rhs = u + dt * (-_convection(u, h, dt) - _grad(p, h) / RHO_F + 0.5 * nu * lap + g)
    lam = 1 + 0.5 * nu * dt * 4 / (h * h) * sum(torch.sin(t) ** 2 for t in _half_angles(n))
    return torch.stack([torch.fft.ifftn(torch.fft.fftn(rhs[c]) / lam).real for c in range(3)])


def _projection(u, p, n, h, dt):
    V = u / dt + _grad(p, h) / RHO_F
    t = _half_angles(n)
    s, c = [torch.sin(x) ** 2 for x in t], [torch.cos(x) ** 2 for x in t]
    lam = -(4 / (h * h)) * (s[0] * c[1] * c[2] + s[1] * c[0] * c[2] + s[2] * c[0] * c[1])
    null = lam.abs() <= 1e-13 * lam.abs().max()
    q = torch.fft.fftn(_div(V, h)) / torch.where(null, torch.ones_like(lam), lam)
    p_new = RHO_F * torch.fft.ifftn(torch.where(null, torch.zeros_like(q), q)).real
    return dt * (V - _grad(p_new, h) / RHO_F), p_new


def _update(parts, n, h, dt, F_ib, T_ib, dIu, dIr):
    X, R, rho = parts["Xr"], parts["radius"], parts["rho_p"]
    V = 4 / 3 * math.pi * R ** 3
    m = rho * V
    L = torch.tensor([k * h for k in n], device=DEV, dtype=F64)
    d = X[None, :, :] - X[:, None, :]
    d = d - L * torch.round(d / L)
    dist = torch.linalg.norm(d, dim=-1)
    Dc = R[:, None] + R[None, :] + h
    near = (dist < Dc) & (dist > 0)
    mean = 0.5 * (m[:, None] + m[None, :])
    k = torch.where(near, -mean * G_COLL / EPS_C * ((dist - Dc) / h) ** 2 / torch.where(dist > 0, dist, torch.ones_like(dist)),
                    torch.zeros_like(dist))
    Fc = (k[:, :, None] * d).sum(1)
    g = torch.tensor(GRAVITY, device=DEV, dtype=F64)
    U = parts["Ur"] + dt / m[:, None] * (F_ib + RHO_F * dIu / dt + (m - RHO_F * V)[:, None] * g + Fc)
    W = parts["Wr"] + dt / (0.4 * m * R * R)[:, None] * (T_ib + RHO_F * dIr / dt)
    return X + 0.5 * dt * (U + parts["Ur"]), U, W


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        out, F, I = [], torch.zeros_like(s["marks"]["R"]), [[], [], []]
        for (a, b), h, f in zip(s["ranges"], s["hs"], s["fields"]):
            off = s["parts"]["moff"][a:b + 1]
            m0, m1 = int(off[0]), int(off[-1])
            parts = {k: v[a:b] for k, v in s["parts"].items() if k != "moff"}
            parts["moff"] = off - m0
            marks = {k: v[m0:m1] for k, v in s["marks"].items()}
            n = (f.shape[3], f.shape[2], f.shape[1])
            u = f.double().reshape(3, -1).clone()
            F[m0:m1] = _forcing(u, n, h, parts, marks, case["Ns"], 1e-3, False, False)
            out.append(u.view(f.shape))
            for k, v in enumerate(_integrals(out[-1], n, h, parts["Xr"], parts["radius"][:, None].expand(-1, 3))):
                I[k].append(v)
        return {"F": F, "I": [torch.cat(v) for v in I], "u": out}
    n, h, dt = s["n"], s["h"], s["dt"]
    u = s["u"].double()
    if kind == "forcing":
        v = u.reshape(3, -1).clone()
        F = _forcing(v, n, h, s["parts"], s["marks"], case["Ns"], dt, case["four"], case["simultaneous"])
        return {"u": v.view(u.shape), "F": F}
    if kind == "transfer":
        idx, wt = _stencil(s["X"], n, h, case["four"])
        f = torch.zeros_like(u).view(3, -1)
        _spread_to(f, idx, wt, s["F"] * (s["marks"]["dV"] / h ** 3)[:, None])
        return {"U": (u.reshape(3, -1)[:, idx] * wt).sum(-1).T, "f": f.view(u.shape)}
    if kind == "integrals":
        ax = s["parts"]["radius"][:, None].expand(-1, 3)
        return {"I0": _integrals(u, n, h, s["parts"]["Xr"], ax), "I1": _integrals(s["u1"].double(), n, h, s["parts"]["Xr"], ax),
                "FT": _force_torque(s["parts"], s["marks"], s["F"])}
    if kind == "ellipsoids":
        return {"I": _integrals(u, n, h, s["Xr"], s["axes"])}
    if kind == "predictor":
        return {"u_star": _predictor(u, s["p"].double(), n, h, case["mu"], dt)}
    if kind == "projection":
        u1, p1 = _projection(u, s["p"].double(), n, h, dt)
        return {"u": u1, "p": p1}
    parts, marks = s["parts"], s["marks"]
    ax = parts["radius"][:, None].expand(-1, 3)
    us = _predictor(u, s["p"].double(), n, h, case["mu"], dt)
    I0 = _integrals(us, n, h, parts["Xr"], ax)
    v = us.reshape(3, -1).clone()
    F = _forcing(v, n, h, parts, marks, case["Ns"], dt, False, False)
    v = v.view(us.shape)
    I1 = _integrals(v, n, h, parts["Xr"], ax)
    F_ib, T_ib = _force_torque(parts, marks, F)
    u1, p1 = _projection(v, s["p"].double(), n, h, dt)
    X, U, W = _update(parts, n, h, dt, F_ib, T_ib, I1[0] - I0[0], I1[1] - I0[1])
    return {"u": u1, "p": p1, "F": F, "Xr": X, "Ur": U, "Wr": W}
