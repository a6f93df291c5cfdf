"""The configuration while a pt_push_stage sequence is open."""
import numpy as np
import pytest
import torch

from paper_2211_05458_gb300 import pt
from paper_2211_05458_gb300 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_the_precision_is_fixed_between_stages(precision):
    """Another precision is refused on the host before anything is launched (the
    state of stage 0 is laid out by it); the sequence goes on unharmed, and the
    precision can be changed after it."""
    wl = W.curved_channel((4, 4, 4), 2, 3, P=500, nsteps=1, dt=2e-3, seed=2)
    ctx = H.gpu_context(wl, precision, schedule=pt.SCHEDULE_STAGED)
    one, stg = H.gpu_particles(wl, ctx), H.gpu_particles(wl, ctx)
    ctx.push(one, 1, wl.dt)
    other = pt.FP64 if precision == "fp32" else pt.FP32
    for s in range(5):
        if s:
            with pytest.raises(pt.PtError) as ei:
                ctx.set_config(precision=other)
            assert ei.value.code == pt.PT_ERR_STATE
            ctx.set_config(max_newton=49)  # the rest of the configuration may change
        ctx.push_stage(stg, s, wl.dt)
    torch.cuda.synchronize()
    a, b = H.gpu_result(one), H.gpu_result(stg)
    for k in ("x", "v", "elem", "hits", "status"):
        assert np.array_equal(a[k], b[k]), k
    ctx.set_config(precision=other)
    assert ctx.precision == other
