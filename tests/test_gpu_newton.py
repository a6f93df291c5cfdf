"""The FP64 inverse map of strongly distorted elements: it converges wherever a
full FP64 Newton iteration from the same trilinear start does, to the same
point."""
import numpy as np
import pytest
import torch

from paper_2211_05458_gb300 import pt
from paper_2211_05458_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _monomials(X, n):
    C = np.linalg.inv(np.vander(np.linspace(-1.0, 1.0, n), n, increasing=True))
    return np.einsum("kc,lb,ma,ecbar->eklmr", C, C, C, X, optimize=True)


def _map(M, xi):
    n = M.shape[1]
    P = [np.stack([xi[:, q] ** k for k in range(n)], 1) for q in range(3)]
    D = [np.stack([k * xi[:, q] ** max(k - 1, 0) for k in range(n)], 1) for q in range(3)]

    def ev(a, b, c):
        return np.einsum("eklmr,ek,el,em->er", M, c, b, a, optimize=True)
    return ev(*P), np.stack([ev(D[0], P[1], P[2]), ev(P[0], D[1], P[2]), ev(P[0], P[1], D[2])], 2)


def _full_newton(M, x, xi, tol=1e-12, maxit=50):
    """As the paper's (Sec. 3.2.1); also the largest condition number of the
    Jacobians met."""
    xi = xi.copy()
    n = len(x)
    ok, live, cond = np.zeros(n, bool), np.ones(n, bool), np.zeros(n)
    for _ in range(maxit):
        i = np.flatnonzero(live)
        if not len(i):
            break
        chi, J = _map(M[i], xi[i])
        cond[i] = np.maximum(cond[i], np.linalg.cond(J))
        d = np.linalg.solve(J, (chi - x[i])[..., None])[..., 0]
        xi[i] -= d
        done = np.abs(d).max(1) < tol
        ok[i[done]] = True
        live[i[done | ~(np.abs(xi[i]).max(1) <= 4.0)]] = False
    return ok, xi, cond


@pytest.mark.parametrize("ngeo,amp", [(2, 0.4), (3, 0.2), (3, 0.3), (4, 0.2), (4, 0.3)])
def test_fp64_inverse_map_of_distorted_elements(ngeo, amp):
    E, n = 20_000 if ngeo < 4 else 10_000, ngeo + 1
    rng = np.random.default_rng(ngeo)
    s = np.linspace(-1.0, 1.0, n)
    c, b, a = np.meshgrid(s, s, s, indexing="ij")
    # every node moved by up to amp of the distance between nodes
    X = np.stack([a, b, c], -1)[None] + amp * (2.0 / ngeo) * rng.uniform(-1, 1, (E, n, n, n, 3))
    M = _monomials(X, n)
    x, _ = _map(M, rng.uniform(-1.0, 1.0, (E, 3)))
    # trilinear start: centre and inverse Jacobian of the corner interpolant
    xc, Jc = _map(_monomials(X[:, ::ngeo, ::ngeo, ::ngeo], 2), np.zeros((E, 3)))
    start = np.linalg.solve(Jc, (x - xc)[..., None])[..., 0].astype(np.float32).astype(float)
    ok, root, cond = _full_newton(M, x, start)
    # the start is formed in FP32 (table and products: up to 1e-6 off), and iterates
    # that wander before they settle depend on its rounding: points whose outcome
    # does not
    use = ok & (cond < 100.0)
    for _ in range(4):
        o, r, _ = _full_newton(M, x, start + 2e-6 * rng.uniform(-1.0, 1.0, (E, 3)))
        use &= o & (np.abs(r - root).max(1) < 1e-9)
    assert use.mean() > 0.9
    none = np.full((E, 6), -1, np.int32)
    mesh = W.Mesh(E, ngeo, X.reshape(E, n ** 3, 3).copy(), none, none.copy(),
                  np.full((E, 6), W.BC_WALL, np.int32), np.zeros((E, 6, 3)))
    ctx = pt.Context(mesh, precision=pt.FP64)
    xi, it, st = ctx.locate(torch.as_tensor(x.T.copy(), device="cuda"),
                            torch.arange(E, dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    xi, st = xi.T.cpu().numpy(), st.cpu().numpy()
    ctx.close()
    lost = np.flatnonzero(use & (st != 0))
    assert lost.size == 0, (lost.size, lost[:5])
    # the last step is below 1e-12 on both sides; a condition number of 100
    # leaves the root itself good to ~1e-13
    assert np.abs(xi - root)[use].max() < 1e-11
