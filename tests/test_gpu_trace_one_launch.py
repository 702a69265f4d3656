"""The trace solve's single launch at the edges of its range: the longest and a short
restart, a system of fewer trace nodes than one CTA's warps, an iteration limit met in
the middle of a cycle; 2D (two blocks per warp step) and 3D.  Against a dense solve."""
import numpy as np
import pytest

from paper_1605_01020_gb300 import workloads as W
from gpu_helpers import dev, host, lib_mesh, rel_err

pytestmark = pytest.mark.gpu


def _system(d, p, cells):
    mesh = W.structured_mesh(d, cells, p)
    field = W.fourier_perturbed_field(2, 0.2, 5) if d == 2 else W.taylor_green_field(0.2)
    st = W.make_state(mesh, field, 7, noise=0.01)
    wl = W.Workload("trace", mesh, st, dict(gamma=1.4, Pr=0.72, Re=1e3, Minf=0.2, alpha=W.dirk_alpha()))
    lm = lib_mesh(wl)
    K, R = lm.assemble_condensed(dev(st.u), dev(st.q), dev(st.uhat))
    rp, col = (host(t).astype(np.int64) for t in lm.trace_pattern())
    A = np.zeros((lm.T, lm.m, lm.T, lm.m))
    r = np.repeat(np.arange(lm.T), np.diff(rp))
    A[r, :, col, :] = host(K)
    return lm, K, R, A.reshape(lm.T * lm.m, -1)


@pytest.mark.parametrize("d,p,cells,restart", [(2, 1, (2, 2), 40), (2, 2, (5, 4), 3), (3, 1, (2, 3, 2), 40), (3, 2, (3, 2, 2), 6)])
def test_restarts_reach_the_dense_solution(d, p, cells, restart):
    lm, K, R, A = _system(d, p, cells)
    dU, its, rr = lm.trace_solve(K, R, restart=restart, max_iter=2000, rtol=1e-12)
    assert rr <= 1e-12 and 0 < its < 2000
    assert rel_err(host(dU), np.linalg.solve(A, host(R).reshape(-1)).reshape(lm.T, lm.m)) <= 1e-8


def test_iteration_limit_inside_a_cycle():
    lm, K, R, A = _system(2, 2, (5, 4))
    dU, its, rr = lm.trace_solve(K, R, restart=4, max_iter=6, rtol=1e-14)
    assert its == 6 and rr > 1e-14
    # the estimate is the true preconditioned residual's (block Jacobi)
    m = lm.m
    x, b = host(dU).reshape(-1), host(R).reshape(-1)
    D = np.stack([A[i * m:(i + 1) * m, i * m:(i + 1) * m] for i in range(lm.T)])
    prec = lambda v: np.linalg.solve(D, v.reshape(lm.T, m, 1)).reshape(-1)
    assert abs(np.linalg.norm(prec(b - A @ x)) / np.linalg.norm(prec(b)) / rr - 1) <= 1e-6
