"""The stage kernel with element slots in shared memory (from 24 particles per
element on, even numbers of nodes) against the resident schedule, which reads
the same data from global memory: the same operations in the same order, so the
results are bitwise equal.  Sizes where the slots can go wrong: the smallest and
largest slot, warps with more owners than slots, particles that have crossed
since the binning, a last warp that is not full."""
import numpy as np
import pytest
import torch

from paper_2211_05458_gb300 import pt
from paper_2211_05458_gb300 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ngeo,N,P", [(1, 1, 27 * 24), (2, 3, 2003), (3, 5, 2500), (4, 5, 1501),
                                      (3, 3, 27 * 64 + 1)])
@pytest.mark.parametrize("mlp", [False, True])
def test_slots_equal_resident(ngeo, N, P, mlp):
    if mlp and ngeo != 3:
        pytest.skip("the learned start needs ngeo = 3")
    wl = W.curved_channel((3, 3, 3), ngeo, N, P=P, nsteps=12, dt=2e-3, seed=ngeo)
    assert P >= 24 * wl.mesh.nelem
    rng = np.random.default_rng(N)
    # few particles in some elements, many in others
    wl.x, wl.elem = W.seed_particles(wl.mesh, P, seed=5, margin=0.2,
                                     elem=(27 * rng.random(P) ** 2).astype(np.int64))
    if ngeo == 1:  # the analytic placement is not inside straight elements
        wl = W.tgv_box(3, N, P, nsteps=12, seed=3, precision="fp32", dt=2e-3)
    wl.v = wl.v * 4.0 + torch.as_tensor(rng.normal(size=tuple(wl.v.shape)) * 1.5)
    net, out = None, []
    for sched in (pt.SCHEDULE_RESIDENT, pt.SCHEDULE_STAGED):
        ctx = H.gpu_context(wl, "fp32", schedule=sched, band_ref=2e-4, band_x=1e-4 / 3)
        if mlp:
            if net is None:
                ctx.mlp_train(*ctx.mlp_make_pairs(20_000, seed=9), epochs=1, batch=1024)
                net = ctx.mlp_get()
            ctx.mlp_set(*net)
            ctx.set_config(guess=pt.GUESS_MLP)
        parts = H.gpu_particles(wl, ctx)
        st = ctx.push(parts, wl.nsteps, wl.dt)
        out.append((H.gpu_result(parts), st))
        ctx.close()
    (a, sa), (b, sb) = out
    assert sa["crossings"] > 0
    for k in ("x", "v", "elem", "hits", "status"):
        assert np.array_equal(a[k], b[k]), k
    assert sa["particle_steps"] == sb["particle_steps"] and sa["crossings"] == sb["crossings"]


def test_state_buffer_follows_the_precision():
    """A context whose precision is switched after a staged push allocates the
    larger FP64 state: the result is a fresh FP64 context's."""
    wl = W.curved_channel((4, 4, 4), 2, 3, P=3001, nsteps=3, dt=2e-3)
    out = []
    for switch in (True, False):
        ctx = H.gpu_context(wl, "fp32" if switch else "fp64", schedule=pt.SCHEDULE_STAGED)
        if switch:
            ctx.push(H.gpu_particles(wl, ctx), 1, wl.dt)
            ctx.set_config(precision=pt.FP64)
            ctx.set_fluid(wl.N, wl.node_type, wl.U.to("cuda", torch.float64).contiguous())
        parts = H.gpu_particles(wl, ctx)
        ctx.push(parts, wl.nsteps, wl.dt)
        out.append(H.gpu_result(parts))
        ctx.close()
    for k in ("x", "v", "elem", "hits", "status"):
        assert np.array_equal(out[0][k], out[1][k]), k
