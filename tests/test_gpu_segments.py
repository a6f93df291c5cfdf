"""The segmented deposition at the edges of its two segment sorts, of its chunks
and of its register tiles, against the one-pass form (bitwise equal)."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2211_05458_gb300 import pt
from paper_2211_05458_gb300 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts", [(0, 1, 2, 31, 32, 33), (64, 65, 127, 128), (129, 130, 700, 0),
                                    (4097, 5, 300, 0)])
@pytest.mark.parametrize("N", [1, 4, 5, 7])
def test_segmented_deposit_of_any_segment_size(counts, N):
    """Segments at the edges of the two sorts and of the 64-particle chunks, and
    every shape of output tile: bitwise the one-pass form's result."""
    nel = len(counts)
    mesh = W.box_mesh((nel, 1, 1), (0.0, 0.0, 0.0), (float(nel), 1.0, 1.0), 2, (False,) * 3)
    el = np.repeat(np.arange(nel), counts)
    np.random.default_rng(0).shuffle(el)
    wl = W.tgv_box(2, N, 4, nsteps=1, precision="fp32")
    wl.mesh, wl.drag_law = mesh, 1
    wl.U = W.fluid_tgv(mesh, N)
    wl.x, wl.elem = W.seed_particles(mesh, len(el), seed=1, elem=el)
    wl.v = torch.zeros_like(wl.x)
    wl.d = torch.full((len(el),), 1e-4, dtype=torch.float64)
    ctx = H.gpu_context(wl, "fp32")
    parts = H.gpu_particles(wl, ctx)
    S = ctx.deposit(parts, pt.DEPOSIT_SEGMENTED)
    T = torch.full_like(S, 7.0)
    p = parts.struct()
    ctx._check(pt.lib().pt_deposit_noalloc(ctx.h, ctypes.byref(p), pt.DEPOSIT_SEGMENTED,
                                           ctypes.c_void_p(T.data_ptr())))
    torch.cuda.synchronize()
    assert torch.equal(S, T)
    assert float(S.abs().max()) > 0.0
