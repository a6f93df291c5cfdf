"""Contexts on a stream of their own that does not wait for the default stream:
the tables that the library copies from the host (mesh, background grid, network,
box list) are there before the kernels that read them, so every result is that of
a context on the default stream."""
import numpy as np
import pytest
import torch

from paper_2211_05458_gb300 import pt
from paper_2211_05458_gb300 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu


def _contexts(make):
    """make() on the default stream and on one that does not wait for it."""
    yield make()
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        yield make()
    torch.cuda.synchronize()


@pytest.mark.parametrize("side,ngeo", [(3, 2), (6, 4), (24, 3)])
def test_mesh_grid_and_push(side, ngeo):
    wl = W.curved_channel((side,) * 3, ngeo, 3, P=5000, nsteps=2, dt=2e-3, seed=1)

    def make():
        ctx = H.gpu_context(wl, "fp32")
        parts = H.gpu_particles(wl, ctx)
        owner, xi, st = ctx.find_element(wl.x.T.contiguous().cuda())
        z, it, ok = ctx.locate(parts.x, parts.elem)
        ctx.push(parts, wl.nsteps, wl.dt)
        out = [t.cpu().numpy() for t in (owner, xi, st, z, ok)] + list(H.gpu_result(parts).values())
        ctx.close()
        return out
    for a, b in zip(*_contexts(make)):
        assert np.array_equal(a, b)


def test_network():
    wl = W.curved_channel((6, 6, 6), 3, 3, P=5000, nsteps=1, dt=2e-3, seed=1)
    first = H.gpu_context(wl, "fp32")
    first.mlp_train(*first.mlp_make_pairs(20_000, seed=9), epochs=1, batch=1024)
    net = first.mlp_get()
    first.close()

    def make():
        ctx = H.gpu_context(wl, "fp32")
        ctx.mlp_set(*net)
        ctx.set_config(guess=pt.GUESS_MLP)
        parts = H.gpu_particles(wl, ctx)
        ctx.push(parts, wl.nsteps, wl.dt)
        out = list(H.gpu_result(parts).values())
        ctx.close()
        return out
    for a, b in zip(*_contexts(make)):
        assert np.array_equal(a, b)


def test_batched_boxes():
    wls = [W.tgv_box(s, N, 700 + s, nsteps=2, seed=s, precision="fp32") for s, N in
           ((3, 3), (5, 4), (4, 3))]

    def make():
        ctxs = [H.gpu_context(wl, "fp32") for wl in wls]
        parts = [H.gpu_particles(wl, c) for wl, c in zip(wls, ctxs)]
        pt.push_batch(ctxs, parts, 2, wls[0].dt)
        out = [v for p in parts for v in H.gpu_result(p).values()]
        for c in ctxs:
            c.close()
        return out
    for a, b in zip(*_contexts(make)):
        assert np.array_equal(a, b)
