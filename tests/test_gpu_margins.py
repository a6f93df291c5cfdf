"""Decisions that the FP32 mode takes in single precision, at the ends of the
ranges that their margins have to cover: long stage displacements in thin
elements that are not aligned with the axes, ends a rounding beyond a wall, and
segments that leave an element by more than its size.  Against the FP64 oracle
or the exact path, particle by particle.  The drag is masked, so that a particle moves on a
straight line and the stage displacements are known beforehand."""
import numpy as np
import pytest
import torch

import oracle
from paper_2211_05458_gb300 import pt
from paper_2211_05458_gb300 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu

B0 = 1432997174477 / 9575080441755  # first stage's share of the step (Carpenter & Kennedy)
DT = 100.0
SCHEDULES = [pt.SCHEDULE_RESIDENT, pt.SCHEDULE_STAGED]


def _workload(mesh, x, elem, v, N=1):
    """One step of particles without forces in a fluid at rest."""
    P = len(elem)
    U = W.fluid_uniform(mesh, N, (0.0, 0.0, 0.0))
    v32 = torch.as_tensor(v, dtype=torch.float32).double()  # what the FP32 mode holds
    return W.Workload("straight", mesh, N, 0, U, torch.as_tensor(x), v32,
                      torch.full((P,), 1e-2, dtype=torch.float64),
                      torch.as_tensor(elem, dtype=torch.int32), 1e-5, 1000.0, 0, DT, 1, "fp32")


def _push(wl, **cfg):
    ctx = H.gpu_context(wl, "fp32", drag_mask=(0.0, 0.0, 0.0), **cfg)
    parts = H.gpu_particles(wl, ctx)
    ctx.push(parts, 1, wl.dt)
    torch.cuda.synchronize()
    g = H.gpu_result(parts)
    ctx.close()
    return g


def _frozen(res):
    return int(((res["status"] & oracle.ST_FROZEN) != 0).sum())


@pytest.mark.parametrize("schedule", SCHEDULES)
@pytest.mark.parametrize("ngeo", [1, 3])
@pytest.mark.parametrize("aspect,length", [(100, 0.2), (300, 0.4), (1000, 0.2), (3000, 0.2)])
def test_long_displacements_in_thin_rotated_elements(aspect, length, ngeo, schedule):
    """Flat elements of the given aspect ratio, rotated, the first stage ending
    1e-6 to 1e-4 (reference units) beyond a face across the thin direction: the
    displacement's long part cancels there.  No particle is lost, each arrives at
    x + dt v and its owner holds it there."""
    P, n = 20_000, (10, 40, 10)
    mesh = W.box_mesh(n, (0.0, 0.0, 0.0), (10.0, 40.0 / aspect, 10.0), ngeo, (False,) * 3)
    rng = np.random.default_rng(aspect + ngeo)
    R = np.linalg.qr(rng.normal(size=(3, 3)))[0]
    mesh.xgeo = mesh.xgeo @ R.T
    ijk = np.stack([rng.integers(4, 6, P), rng.integers(12, 28, P), rng.integers(4, 6, P)], 1)
    elem = ijk[:, 0] + n[0] * (ijk[:, 1] + n[1] * ijk[:, 2])
    h = np.array([1.0, 1.0 / aspect, 1.0])
    xi = rng.uniform(-0.9, 0.9, (P, 3))
    y = (ijk + 0.5 * (xi + 1.0)) * h
    phi = rng.uniform(0.0, 2.0 * np.pi, P)
    side = rng.choice([-1.0, 1.0], P)
    end = side * (1.0 + 10.0 ** rng.uniform(-6.0, -4.0, P))
    dy = np.stack([length * np.cos(phi), 0.5 * h[1] * (end - xi[:, 1]), length * np.sin(phi)], 1)
    wl = _workload(mesh, y @ R.T, elem, (dy / (B0 * DT)) @ R.T)
    g = _push(wl, schedule=schedule)
    assert _frozen(g) == 0 and int(g["hits"].sum()) == 0
    # five increments of at most the whole path, each with a few FP32 roundings
    x1 = (wl.x + DT * wl.v).numpy()
    assert np.abs(g["x"] - x1).max() <= 30 * 6e-8 * length / B0
    e = g["elem"]
    own = np.stack([e % n[0], e // n[0] % n[1], e // (n[0] * n[1])], 1)
    z = 2.0 * ((g["x"] @ R) / h - own) - 1.0
    assert np.abs(z).max() <= 1.0 + 1e-6  # lost_tol


@pytest.mark.parametrize("schedule", SCHEDULES)
@pytest.mark.parametrize("ngeo", [1, 2])
@pytest.mark.parametrize("length", [0.05, 0.2, 0.4, 0.9])
def test_ends_a_rounding_beyond_a_wall(length, ngeo, schedule):
    """Unit cubes, the first stage ending 0 to 1e-7 beyond a wall: it is
    reflected there or, if the end is taken as inside, at the next stage's
    start, and never lost."""
    P = 20_000
    mesh = W.box_mesh((3, 3, 3), (0.0, 0.0, 0.0), (3.0, 3.0, 3.0), ngeo, (False,) * 3)
    rng = np.random.default_rng(int(100 * length) + ngeo)
    jk = rng.integers(0, 3, (P, 2))
    elem = 2 + 3 * (jk[:, 0] + 3 * jk[:, 1])
    cos = rng.uniform(0.5, 1.0, P)
    phi = rng.uniform(0.0, 2.0 * np.pi, P)
    t = np.sqrt(1.0 - cos * cos)
    dx = length * np.stack([cos, t * np.cos(phi), t * np.sin(phi)], 1)
    v = (dx / (B0 * DT)).astype(np.float32)
    # the displacement as the FP32 mode forms it
    d1 = (np.float32(B0) * (np.float32(DT) * v[:, 0])).astype(np.float64)
    x = np.stack([3.0 + rng.uniform(0.0, 1e-7, P) - d1, jk[:, 0] + rng.uniform(0.05, 0.95, P),
                  jk[:, 1] + rng.uniform(0.05, 0.95, P)], 1)
    wl = _workload(mesh, x, elem, v)
    o = H.run_oracle(wl, mask=(0.0, 0.0, 0.0))
    assert _frozen(o) == 0 and int((o["hits"] > 0).sum()) == P
    g = _push(wl, schedule=schedule)
    assert _frozen(g) == 0
    assert np.array_equal(g["hits"], o["hits"])
    assert np.abs(g["x"] - o["x"]).max() <= 30 * 6e-8 * length / B0


@pytest.mark.parametrize("schedule", SCHEDULES)
@pytest.mark.parametrize("ngeo,c,reach", [(4, 0.0035, 2.5), (4, 0.004, 2.4), (4, 0.003, 2.7),
                                          (4, 0.01, 1.5), (3, 0.01, 2.5), (2, 0.02, 2.0)])
def test_segments_that_leave_the_element_far_behind(ngeo, c, reach, schedule):
    """Elements stretched along x by xi + c (xi^p - 1 or xi), first stages from
    within band_x of the wall at x = 0 to xi = reach in the first element's
    extended map, where its curvature is far above that inside: the wall that
    the segment starts at still counts as met (PT_ST_NEAR_WALL)."""
    P, nx, band = 2000, 24, 1e-3
    odd = ngeo % 2 == 1
    g1 = (lambda s: s + c * (s ** ngeo - s)) if odd else (lambda s: s + c * (s ** ngeo - 1.0))
    mesh = W.box_mesh((nx, 2, 2), (0.0, 0.0, 0.0), (float(nx), 2.0, 2.0), ngeo, (False,) * 3)
    s = np.linspace(-1.0, 1.0, ngeo + 1)
    i = np.arange(mesh.nelem) % nx
    X = mesh.xgeo.reshape(mesh.nelem, -1, ngeo + 1, 3)  # (xi1 fastest)
    X[..., 0] = i[:, None, None] + 0.5 * (1.0 + g1(s))[None, None, :]
    rng = np.random.default_rng(ngeo)
    jk = rng.integers(0, 2, (P, 2))
    elem = nx * (jk[:, 0] + 2 * jk[:, 1])
    x = np.stack([rng.uniform(0.1, 0.8, P) * band, jk[:, 0] + rng.uniform(0.4, 0.6, P),
                  jk[:, 1] + rng.uniform(0.4, 0.6, P)], 1)
    dx = np.zeros((P, 3))
    dx[:, 0] = 0.5 * (1.0 + g1(reach)) - x[:, 0]
    wl = _workload(mesh, x, elem, dx / (B0 * DT))
    o = H.run_oracle(wl, band_x=band, mask=(0.0, 0.0, 0.0))
    assert _frozen(o) == 0 and bool((o["status"] & oracle.ST_NEAR_WALL).all())
    g = _push(wl, schedule=schedule, band_x=band)
    assert _frozen(g) == 0 and np.array_equal(g["elem"], o["elem"])
    missed = (g["status"] & oracle.ST_NEAR_WALL) == 0
    assert not missed.any(), int(missed.sum())


@pytest.mark.parametrize("ngeo", [2, 3, 4])
def test_large_steps_between_curved_walls(ngeo):
    """Stage displacements up to about an element between curved walls: owners,
    wall hits, states and positions are those of the FP64 mode, which intersects
    every face in FP64."""
    mesh = W.channel_mesh((6, 5, 4), ngeo, amp=0.1, curved_walls=True)
    P = 600
    wl = W.curved_channel((6, 5, 4), ngeo, 3, P=P, nsteps=2, dt=0.15, seed=ngeo)
    wl.mesh = mesh
    wl.U, _ = W.fluid_channel(mesh, 3, 0, seed=0)
    wl.x, wl.elem = W.seed_particles(mesh, P, seed=ngeo)
    rng = np.random.default_rng(ngeo)
    wl.v = torch.as_tensor(rng.normal(size=(P, 3)) * np.array([6.0, 3.0, 4.0]))
    wl.v = wl.v.float().double()
    wl.d = torch.full((P,), 2e-2, dtype=torch.float64)  # Stokes number 2200: nearly straight
    band = dict(band_ref=2e-4, band_x=4e-5)
    out = []
    for precision in ("fp32", "fp64"):
        ctx = H.gpu_context(wl, precision, **band)
        parts = H.gpu_particles(wl, ctx)
        ctx.push(parts, wl.nsteps, wl.dt)
        torch.cuda.synchronize()
        out.append(H.gpu_result(parts))
        ctx.close()
    ref = out[1]
    assert int(ref["hits"].sum()) > P // 4
    ref["_orc"], ref["_params"] = H.make_oracle(wl), H.oracle_params(wl, **band)
    H.compare(out[0], ref, 2e-5, min_checked=0.85)
