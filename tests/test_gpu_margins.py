"""Decisions that the FP32 mode takes in single precision, at the ends of the
ranges that their margins have to cover: long stage displacements in thin
elements that are not aligned with the axes and ends a rounding beyond a wall.
Against the FP64 oracle
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
