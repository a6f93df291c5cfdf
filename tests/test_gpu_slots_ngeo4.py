"""Element slots at NGeo = 4, whose rows of six coefficients are read in pairs:
the stage kernel with slots (N = 1 and 3 fit, from 24 particles per element on)
against the resident schedule, bitwise as the same operations run in the same
order; N = 5 does not fit and takes the kernel without slots."""
import numpy as np
import pytest
import torch

from paper_2211_05458_gb300 import pt
from paper_2211_05458_gb300 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,P", [(1, 27 * 24), (1, 2003), (3, 27 * 24 + 1), (3, 2500), (5, 1501)])
def test_ngeo4_slots_equal_resident(N, P):
    wl = W.curved_channel((3, 3, 3), 4, N, P=P, nsteps=12, dt=2e-3, seed=4)
    rng = np.random.default_rng(P)
    # few particles in some elements, many in others; starts close to the faces
    wl.x, wl.elem = W.seed_particles(wl.mesh, P, seed=6, margin=0.01,
                                     elem=(27 * rng.random(P) ** 2).astype(np.int64))
    wl.v = wl.v * 4.0 + torch.as_tensor(rng.normal(size=tuple(wl.v.shape)) * 1.5)
    out = []
    for sched in (pt.SCHEDULE_RESIDENT, pt.SCHEDULE_STAGED):
        ctx = H.gpu_context(wl, "fp32", schedule=sched, band_ref=2e-4, band_x=1e-4 / 3)
        parts = H.gpu_particles(wl, ctx)
        st = ctx.push(parts, wl.nsteps, wl.dt)
        out.append((H.gpu_result(parts), st))
        ctx.close()
    (a, sa), (b, sb) = out
    assert sa["crossings"] > 0
    for k in ("x", "v", "elem", "hits", "status"):
        assert np.array_equal(a[k], b[k]), k
    assert sa["particle_steps"] == sb["particle_steps"] and sa["crossings"] == sb["crossings"]
