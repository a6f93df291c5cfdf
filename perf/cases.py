"""The work that is timed: calls of a particle push in a flow solver's time loop.

A case is one call (or one short sequence of calls) of the public API on a mesh,
a fluid state and a particle set.  A flow solver that advances the fluid every
time step calls the push with one or a few steps at a time, so most cases run
1 to 10 steps per pass; the particle arrays are updated in place and the next
pass goes on from there.

In PT_FP32 mode the near-face bands are set to what single precision resolves
(band_ref 2e-4, band_x 1e-4 of an element), as the parity tests do: with the
1e-10 default a status bit there tells rounding, not position.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2211_05458_gb300 import pt
from paper_2211_05458_gb300 import workloads as W

DEV = "cuda"

# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------


def _push(name, dims, ngeo, N, P, steps, prec="fp32", box=False, drag=1, guess="trilinear",
          track="physical", call="push", gravity=False, dt=1e-3, nodes=0):
    return dict(name=name, kind="push", nx=dims[0], ny=dims[1], nz=dims[2], ngeo=ngeo, N=N, P=P,
                steps=steps, prec=prec, box=box, drag=drag, guess=guess, track=track, call=call,
                gravity=gravity, dt=dt, nodes=nodes)


def listed():
    return [
        # the smallest call: one step of a thousand particles, launch latency
        _push("few_particles_one_step", (8, 8, 8), 2, 3, 1000, 1),
        # the small FP64 configuration: straight 8^3 box, Stokes drag, 10^4 particles at rest
        _push("box_fp64_1e4", (8, 8, 8), 1, 3, 10_000, 10, prec="fp64", box=True, drag=0),
        # an ordinary FP32 call below the size where the library changes its
        # schedule: ragged mesh, odd degree and count, Gauss-Lobatto nodes
        _push("channel_fp32_ragged", (13, 17, 11), 3, 4, 100_003, 2, nodes=1),
        # the 32^3 channel of 10^6 particles in both precisions
        _push("channel_fp64_1e6", (32, 32, 32), 2, 5, 1_000_000, 1, prec="fp64"),
        _push("channel_fp32_1e6", (32, 32, 32), 2, 5, 1_000_000, 3),
        # the learned-start configuration (64^3, 10^7 particles) at its particles
        # per element on a mesh that is set up in a few seconds
        _push("channel_learned_4e6", (48, 48, 48), 3, 5, 4_200_000, 2, guess="mlp"),
        # localisation in reference space, gravity with buoyancy, NGeo = 4
        _push("channel_reference_gravity", (24, 20, 18), 4, 6, 700_001, 2, track="reference",
              gravity=True),
        # a solver that calls the push once per Runge-Kutta stage
        _push("channel_stage_calls", (24, 24, 24), 2, 3, 500_000, 1, call="stage"),
        # a caller whose particles live in (pinned) host memory
        _push("channel_host_arrays", (24, 24, 24), 2, 5, 1_000_000, 2, call="host"),
        # many independent boxes of uneven size in one call
        dict(name="boxes_16", kind="boxes", nbox=16, layout=1, side_lo=8, side_hi=24, P_lo=1000,
             P_hi=300_000, steps=5, dt=1e-3),
        # two-way coupling: one step and the deposition of the drag on the nodes
        dict(name="two_way_segmented", kind="deposit", nx=64, ny=32, nz=32, ngeo=2, N=7,
             P=2_500_000, steps=1, mode="segmented", nearest=False, prec="fp32", dt=1e-3),
        # initial placement: which element owns each point
        dict(name="find_owner_1e6", kind="find", nx=32, ny=32, nz=32, ngeo=3, P=1_000_000,
             prec="fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dims(rng, lo=5, hi=36):
    """Mesh sizes of like extent per direction, odd ones among them."""
    m = _log_int(rng, lo, hi)
    return tuple(max(3, min(hi, m + rng.randint(-m // 4, m // 4))) for _ in range(3))


def draw(rng):
    kind = rng.choice(["push", "push", "push", "push", "deposit", "boxes", "find"])
    if kind == "push":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        ngeo = rng.randint(1, 4)
        P = _log_int(rng, 500, 1_000_000 if prec == "fp32" else 300_000)
        steps = rng.randint(1, 3 if P > 200_000 else 5)
        call = rng.choice(["push", "push", "push", "stage", "host"])
        guess = "mlp" if ngeo == 3 and prec == "fp32" and rng.random() < 0.5 else "trilinear"
        box = ngeo == 1 and rng.random() < 0.5
        c = _push("", _dims(rng), ngeo, rng.randint(1, 7), P, 1 if call == "stage" else steps,
                  prec=prec, box=box, drag=0 if box else 1, guess=guess, call=call,
                  track="reference" if rng.random() < 0.2 else "physical",
                  gravity=rng.random() < 0.2, nodes=rng.randint(0, 1))
    elif kind == "deposit":
        nx, ny, nz = _dims(rng, 5, 32)
        c = dict(name="", kind="deposit", nx=nx, ny=ny, nz=nz, ngeo=rng.randint(1, 4),
                 N=rng.randint(1, 7), P=_log_int(rng, 1000, 1_000_000), steps=rng.randint(0, 1),
                 mode=rng.choice(["segmented", "segmented", "atomic"]),
                 nearest=rng.random() < 0.25, prec=rng.choice(["fp32", "fp32", "fp64"]), dt=1e-3)
    elif kind == "boxes":
        c = dict(name="", kind="boxes", nbox=rng.randint(2, 24), layout=rng.randint(2, 10_000),
                 side_lo=6, side_hi=rng.randint(10, 24), P_lo=1000,
                 P_hi=_log_int(rng, 20_000, 200_000), steps=rng.randint(1, 5), dt=1e-3)
    else:
        nx, ny, nz = _dims(rng)
        c = dict(name="", kind="find", nx=nx, ny=ny, nz=nz, ngeo=rng.randint(1, 4),
                 P=_log_int(rng, 1000, 1_000_000), prec=rng.choice(["fp32", "fp64"]))
    del c["name"]
    return c


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------


@functools.lru_cache(maxsize=4)
def _mesh(dims, ngeo, box):
    if box:
        return W.box_mesh(dims, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), ngeo)
    return W.channel_mesh(dims, ngeo)


def _lagrange(nodes):
    """Monomial coefficients C[a, k] of the Lagrange basis on nodes."""
    n = len(nodes)
    C = np.zeros((n, n))
    for a in range(n):
        p = np.poly1d([1.0])
        for m in range(n):
            if m != a:
                p = p * np.poly1d([1.0, -nodes[m]]) / (nodes[a] - nodes[m])
        C[a, :len(p.coeffs)] = p.coeffs[::-1]
    return torch.tensor(C, device=DEV)


def _powers(x, n):
    """[..., n] powers 0 .. n-1 of x, and their derivatives."""
    p = [torch.ones_like(x)]
    for _ in range(n - 1):
        p.append(p[-1] * x)
    d = [torch.zeros_like(x)] + [k * p[k - 1] for k in range(1, n)]
    return torch.stack(p, dim=-1), torch.stack(d, dim=-1)


def _solve(J, r):
    """J^-1 r for [n, 3, 3] and [n, 3] by cross products."""
    a, b, c = J[:, :, 0], J[:, :, 1], J[:, :, 2]
    bc = torch.linalg.cross(b, c)
    det = (a * bc).sum(dim=1, keepdim=True)
    return torch.stack([(r * bc).sum(dim=1), (r * torch.linalg.cross(c, a)).sum(dim=1),
                        (r * torch.linalg.cross(a, b)).sum(dim=1)], dim=1) / det


class _Map:
    """The element map of a mesh in 64 bits."""

    def __init__(self, mesh):
        self.g = mesh.ngeo + 1
        self.X = torch.tensor(mesh.xgeo, device=DEV).reshape(mesh.nelem, self.g, self.g, self.g, 3)
        self.C = _lagrange(np.linspace(-1.0, 1.0, self.g))
        self.nbr = torch.tensor(mesh.neighbor, device=DEV).long()
        self.bc = torch.tensor(mesh.bc, device=DEV)
        self.shift = torch.tensor(mesh.shift, device=DEV)

    def at(self, e, xi, jac=False):
        P, D = _powers(xi, self.g)
        l, dl = P @ self.C.T, D @ self.C.T
        A = self.X[e]  # [n, c, b, a, 3]
        T = torch.einsum("ncbar,na->ncbr", A, l[:, 0])
        V = torch.einsum("ncbr,nb->ncr", T, l[:, 1])
        x = torch.einsum("ncr,nc->nr", V, l[:, 2])
        if not jac:
            return x
        T1 = torch.einsum("ncbar,na->ncbr", A, dl[:, 0])
        j0 = torch.einsum("ncbr,nb,nc->nr", T1, l[:, 1], l[:, 2])
        j1 = torch.einsum("ncbr,nb,nc->nr", T, dl[:, 1], l[:, 2])
        j2 = torch.einsum("ncr,nc->nr", V, dl[:, 2])
        return x, torch.stack([j0, j1, j2], dim=-1)

    def inverse(self, e, x, xi=None):
        xi = torch.zeros_like(x) if xi is None else xi.clone()
        for _ in range(12):
            y, J = self.at(e, xi, True)
            d = _solve(J, x - y)
            xi = xi + d
            if float(d.abs().max()) < 1e-13:
                break
        return xi


def _config(case, mesh):
    cfg = dict(precision=pt.FP64 if case["prec"] == "fp64" else pt.FP32)
    if case["prec"] == "fp32":
        cfg.update(band_ref=2e-4, band_x=1e-4 * (mesh.hi[1] - mesh.lo[1]) / mesh.dims[1])
    if case.get("track") == "reference":
        cfg["track"] = pt.TRACK_REFERENCE
    if case.get("gravity"):
        cfg.update(g=(0.0, -9.81, 0.0), buoyancy=1)
    cfg["drag_law"] = case.get("drag", 1)
    return cfg


def _placed(mesh, P, seed):
    """P points drawn uniformly in reference space: owner, reference position, x."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    e = torch.randint(0, mesh.nelem, (P,), generator=gen, device=DEV)
    xi = (torch.rand((P, 3), generator=gen, dtype=torch.float64, device=DEV) * 2.0 - 1.0) * 0.99
    m = _Map(mesh)
    x = torch.cat([m.at(e[i:i + 250_000], xi[i:i + 250_000]) for i in range(0, P, 250_000)])
    return e, xi, x


def _inputs(case, seed):
    """Mesh, fluid state and particles of a push, as the library is given them."""
    dims = (case["nx"], case["ny"], case["nz"])
    mesh = _mesh(dims, case["ngeo"], case.get("box", False))
    real = torch.float64 if case["prec"] == "fp64" else torch.float32
    P, N, nodes = case["P"], case["N"], case.get("nodes", 0)
    e, _, x = _placed(mesh, P, seed)
    if case.get("box"):
        # a Taylor-Green vortex on a mean flow drawn from the seed, particles at rest
        U = W.fluid_tgv(mesh, N, nodes, DEV)
        w = torch.tensor(np.random.default_rng(seed).uniform(-0.2, 0.2, 3), device=DEV)
        U[:, 1:4] += U[:, 0:1] * w.view(1, 3, 1)
        v = torch.zeros_like(x)
        d = torch.full((P,), 1e-4, dtype=torch.float64, device=DEV)
    else:
        # channel turbulence, particles at the fluid velocity with a spread
        U, scale = W.fluid_channel(mesh, N, nodes, seed % 100_003, DEV)
        u = W.channel_velocity(x[:, 0], x[:, 1], x[:, 2], seed=seed % 100_003, scale=scale)
        gen = torch.Generator(device=DEV).manual_seed(seed + 17)
        v = torch.stack(u[:3], dim=1) + 0.05 * torch.randn((P, 3), generator=gen, device=DEV,
                                                           dtype=torch.float64)
        # Stokes numbers log-uniform in [0.1, 100]
        tau = 0.1 * 1000.0 ** torch.rand(P, generator=gen, device=DEV, dtype=torch.float64)
        d = torch.sqrt(18.0 * 1e-5 * tau / 1000.0)
    return mesh, U.to(real).contiguous(), x, v.to(real), d.to(real), e.to(torch.int32)


def _boxes(case, seed):
    """(side, N, P, background flow) of each box: sides, degrees and counts from
    the layout, the flow and the particles from the seed."""
    rng = np.random.default_rng(case["layout"])
    flow = np.random.default_rng(seed)
    out = []
    for _ in range(case["nbox"]):
        side = int(round(math.exp(rng.uniform(math.log(case["side_lo"]),
                                              math.log(case["side_hi"])))))
        N = int(rng.integers(3, 8))
        P = int(round(math.exp(rng.uniform(math.log(case["P_lo"]), math.log(case["P_hi"])))))
        out.append((side, N, P, int(flow.integers(1 << 30))))
    return out


def _box_case(b, case):
    return dict(nx=b[0], ny=b[0], nz=b[0], ngeo=1, N=b[1], P=b[2], prec="fp32", box=True,
                drag=0, steps=case["steps"], dt=case["dt"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "find":
        mesh = _mesh((case["nx"], case["ny"], case["nz"]), case["ngeo"], False)
        ctx = pt.Context(mesh, **_config(case, mesh))
        _, _, x = _placed(mesh, case["P"], seed)
        x = x.T.contiguous()
        ctx.find_element(x[:, :1].contiguous())  # the background grid is kept by the context
        return dict(kind=kind, ctx=ctx, x=x)
    if kind == "boxes":
        ctxs, parts = [], []
        for b in _boxes(case, seed):
            c = _box_case(b, case)
            mesh, U, x, v, d, e = _inputs(c, b[3])
            ctx = pt.Context(mesh, **_config(c, mesh))
            ctx.set_fluid(b[1], 0, U)
            ctxs.append(ctx)
            parts.append(pt.ParticleSet.create(x, v, d, e, pt.FP32, DEV))
        return dict(kind=kind, ctxs=ctxs, parts=parts, steps=case["steps"], dt=case["dt"])
    mesh, U, x, v, d, e = _inputs(case, seed)
    ctx = pt.Context(mesh, **_config(case, mesh))
    ctx.set_fluid(case["N"], case.get("nodes", 0), U)
    if case.get("guess") == "mlp":
        pairs = ctx.mlp_make_pairs(100_000, seed=3)
        ctx.mlp_train(*pairs, epochs=2, batch=1024, lr=2e-3, seed=0)
        ctx.set_config(guess=pt.GUESS_MLP)
    host = case.get("call") == "host"
    parts = pt.ParticleSet.create(x, v, d, e, ctx.precision, "cpu" if host else DEV, pin=host)
    s = dict(kind=kind, ctx=ctx, parts=parts, steps=case["steps"], dt=case["dt"],
             call=case.get("call", "push"))
    if kind == "deposit":
        s["mode"] = ((pt.DEPOSIT_SEGMENTED if case["mode"] == "segmented" else pt.DEPOSIT_ATOMIC)
                     | (pt.DEPOSIT_NEAREST if case["nearest"] else 0))
        s["S"] = torch.empty((mesh.nelem, 4, (case["N"] + 1) ** 3), dtype=torch.float32,
                             device=DEV)
    return s


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------


def _state(p):
    return dict(x=p.x, v=p.v, elem=p.elem, hits=p.hits, status=p.status)


def run(s):
    if s["kind"] == "find":
        elem, xi, status = s["ctx"].find_element(s["x"])
        return dict(elem=elem, xi=xi, status=status)
    if s["kind"] == "boxes":
        pt.push_batch(s["ctxs"], s["parts"], s["steps"], s["dt"], stats=False)
        # the boxes' arrays joined: one output per quantity
        return {k: torch.cat([getattr(p, k).reshape(-1) for p in s["parts"]])
                for k in ("x", "v", "elem", "hits", "status")}
    ctx, parts = s["ctx"], s["parts"]
    if s["call"] == "host":
        ctx.push_host(parts, s["steps"], s["dt"], stats=False)
    elif s["call"] == "stage":
        for _ in range(s["steps"]):
            for stage in range(5):
                ctx.push_stage(parts, stage, s["dt"])
    elif s["steps"]:
        ctx.push(parts, s["steps"], s["dt"], stats=False)
    out = _state(parts)
    if s["kind"] == "deposit":
        out["S"] = ctx.deposit(parts, s["mode"], s["S"])
    return out


# ----------------------------------------------------------------------------
# work of one pass
# ----------------------------------------------------------------------------


def _push_work(c):
    """Particle state in and out, each element's nodes and rho, rho u once; the
    flops of two Newton steps (map and Jacobian), the interpolation and the rest
    of a stage, sum-factorised."""
    r = 8 if c["prec"] == "fp64" else 4
    g, n, E = c["ngeo"] + 1, c["N"] + 1, min(c["nx"] * c["ny"] * c["nz"], c["P"])
    part = (24 + 3 * r + r + 12) + (24 + 3 * r + 12)
    newton = 3 * (2 * (2 * g ** 3 + 3 * g * g + 4 * g)) + 60
    interp = 4 * 2 * (n ** 3 + n * n + n) + 3 * 6 * n
    return (c["P"] * part + E * (4 * n ** 3 * r + 3 * g ** 3 * r),
            c["P"] * 5.0 * c["steps"] * (2 * newton + interp + 150))


def work(case):
    if case["kind"] == "boxes":
        w = [_push_work(_box_case(b, case)) for b in _boxes(case, 0)]
        return dict(bytes=float(sum(x[0] for x in w)), flops=float(sum(x[1] for x in w)))
    g = case["ngeo"] + 1
    E = min(case["nx"] * case["ny"] * case["nz"], case["P"])
    newton = 3 * (2 * (2 * g ** 3 + 3 * g * g + 4 * g)) + 60
    if case["kind"] == "find":
        r = 8 if case["prec"] == "fp64" else 4
        return dict(bytes=float(case["P"] * (24 + 4 + 24 + 4) + E * 3 * g ** 3 * r),
                    flops=float(case["P"] * 3 * newton))
    b, f = _push_work(case)
    if case["kind"] == "deposit":
        r = 8 if case["prec"] == "fp64" else 4
        n = case["N"] + 1
        if not case["steps"]:
            b = case["P"] * (24 + 4 * r + 8) + E * (4 * n ** 3 * r + 3 * g ** 3 * r)
        b += 16 * n ** 3 * case["nx"] * case["ny"] * case["nz"]
        spread = 8 * (4 if case["nearest"] else n ** 3 + 2 * n * n)
        f += case["P"] * (2 * newton + 4 * 2 * (n ** 3 + n * n + n) + spread)
    return dict(bytes=float(b), flops=float(f))


# ----------------------------------------------------------------------------
# the same in 64 bits with plain torch
# ----------------------------------------------------------------------------

# Carpenter & Kennedy (1994), five-stage fourth-order 2N-storage scheme
RK_A = [0.0, -567301805773.0 / 1357537059087.0, -2404267990393.0 / 2016746695238.0,
        -3550918686646.0 / 2091501179385.0, -1275806237668.0 / 842570457699.0]
RK_B = [1432997174477.0 / 9575080441755.0, 5161836677717.0 / 13612068292357.0,
        1720146321549.0 / 2090206949498.0, 3134564353537.0 / 4481467310338.0,
        2277821191437.0 / 14882151754819.0]
MU, RHO_P = 1e-5, 1000.0


def _interp(U, C, e, xi):
    n = C.shape[0]
    P, _ = _powers(xi, n)
    l = P @ C.T
    A = U[e, :4].double().reshape(-1, 4, n, n, n)
    t = torch.einsum("nvcba,na->nvcb", A, l[:, 0])
    return torch.einsum("nvcb,nb,nc->nv", t, l[:, 1], l[:, 2]), l


def _factor(case, Uv, rel, d):
    if case.get("drag", 1) == 0:
        return torch.ones_like(d)
    return 1.0 + 0.15 * (Uv[:, 0] * rel.norm(dim=1) * d / MU) ** 0.687


def _exact_push(case, mesh, m, C, U, x, v, d, e):
    """Stages of the push: the owner of a stage's end is found by the inverse
    map and a walk over the faces; walls are the planes y = lo, hi."""
    g = torch.tensor([0.0, -9.81 if case.get("gravity") else 0.0, 0.0], device=DEV,
                     dtype=torch.float64)
    tau = RHO_P * d * d / (18.0 * MU)
    walls = not case.get("box", False)
    for _ in range(case["steps"]):
        kx, kv = torch.zeros_like(x), torch.zeros_like(v)
        for s in range(5):
            xi = m.inverse(e, x)
            Uv, _ = _interp(U, C, e, xi)
            rel = Uv[:, 1:4] / Uv[:, :1] - v
            a = (_factor(case, Uv, rel, d) / tau)[:, None] * rel
            a = a + g * ((1.0 - Uv[:, :1] / RHO_P) if case.get("gravity") else 1.0)
            kx = RK_A[s] * kx + case["dt"] * v
            kv = RK_A[s] * kv + case["dt"] * a
            x = x + RK_B[s] * kx
            v = v + RK_B[s] * kv
            if walls:
                for y, sgn in ((mesh.hi[1], 1.0), (mesh.lo[1], -1.0)):
                    hit = sgn * (x[:, 1] - y) > 0.0
                    x[:, 1] = torch.where(hit, 2.0 * y - x[:, 1], x[:, 1])
                    for q in (v, kx, kv):
                        q[:, 1] = torch.where(hit, -q[:, 1], q[:, 1])
            todo = torch.arange(len(e), device=DEV)
            e = e.clone()
            for _ in range(6):
                z = m.inverse(e[todo], x[todo])
                out = z.abs().max(dim=1)[0] > 1.0
                if not bool(out.any()):
                    break
                todo, z = todo[out], z[out]
                q = z.abs().argmax(dim=1)
                f = 2 * q + (z.gather(1, q[:, None])[:, 0] > 0).long()
                et = e[todo]
                nb = m.nbr[et, f]
                inside = nb >= 0
                x[todo] += m.shift[et, f] * inside[:, None]
                e[todo] = torch.where(inside, nb, et)
    return x, v, e


def _exact_deposit(case, m, C, U, x, v, d, e):
    n = C.shape[0]
    xi = m.inverse(e, x)
    Uv, l = _interp(U, C, e, xi)
    rel = Uv[:, 1:4] / Uv[:, :1] - v
    F = (3.0 * math.pi * MU * d * _factor(case, Uv, rel, d))[:, None] * rel
    f = torch.cat([-F, -(F * v).sum(dim=1, keepdim=True)], dim=1)
    if not case["nearest"]:
        return torch.einsum("nq,nc,nb,na->nqcba", f, l[:, 2], l[:, 1], l[:, 0]).reshape(
            len(e), 4, n ** 3)
    sn, sw = np.polynomial.legendre.leggauss(n)
    sn, sw = torch.tensor(sn, device=DEV), torch.tensor(sw, device=DEV)
    q = (xi[:, :, None] - sn).abs().argmin(dim=2)
    _, J = m.at(e, sn[q], True)
    f = f / (sw[q].prod(dim=1) * torch.linalg.det(J).abs())[:, None]
    w = torch.zeros((len(e), n ** 3), dtype=torch.float64, device=DEV)
    w.scatter_(1, (q[:, 0] + n * (q[:, 1] + n * q[:, 2]))[:, None], 1.0)
    return f[:, :, None] * w[:, None, :]


def _exact_one(case, inputs):
    mesh, U, x, v, d, e = inputs
    m = _Map(mesh)
    n = case["N"] + 1
    C = _lagrange(W.solution_nodes(case["N"], case.get("nodes", 0)))
    S = (torch.zeros((mesh.nelem, 4, n ** 3), dtype=torch.float64, device=DEV)
         if case.get("kind") == "deposit" else None)
    xs, vs = [], []
    chunk = 200_000 if S is None else max(2000, 20_000_000 // n ** 3)
    for i in range(0, len(e), chunk):
        q = slice(i, i + chunk)
        xq, vq, dq, eq = x[q].clone(), v[q].double(), d[q].double(), e[q].long()
        xq, vq, eq = _exact_push(case, mesh, m, C, U, xq, vq, dq, eq)
        if S is not None:
            S.index_add_(0, eq, _exact_deposit(case, m, C, U, xq, vq, dq, eq))
        xs.append(xq)
        vs.append(vq)
    return torch.cat(xs).T.contiguous(), torch.cat(vs).T.contiguous(), S


def exact(case, seed):
    """Positions, velocities, sources and reference positions; owners, hit
    counts and status bits are whole numbers and have no value here."""
    if case["kind"] == "find":
        mesh = _mesh((case["nx"], case["ny"], case["nz"]), case["ngeo"], False)
        return dict(elem=None, xi=_placed(mesh, case["P"], seed)[1].T.contiguous(), status=None)
    if case["kind"] == "boxes":
        got = []
        for b in _boxes(case, seed):
            c = _box_case(b, case)
            got.append(_exact_one(c, _inputs(c, b[3])))
        return dict(x=torch.cat([q[0].reshape(-1) for q in got]),
                    v=torch.cat([q[1].reshape(-1) for q in got]), elem=None, hits=None,
                    status=None)
    x, v, S = _exact_one(case, _inputs(case, seed))
    out = dict(x=x, v=v, elem=None, hits=None, status=None)
    if case["kind"] == "deposit":
        out["S"] = S
    return out
