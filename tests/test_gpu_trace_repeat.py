"""The trace solve's sums over the grid belong to one reduction each: a thousand solves of
one system give the same bits and step counts.  (A partial sum that the next reduction
overwrites before every block has read it shows as a solve that differs; the smallest
systems, with few rows a block, leave the least time between the two.)"""
import pytest

from paper_1605_01020_gb300 import workloads as W
from gpu_helpers import dev, lib_mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,p,cells,solves", [(2, 2, (8, 8), 1000), (3, 3, (6, 6, 6), 1000), (2, 1, (3, 2), 1000)])
def test_solves_repeat_bit_for_bit(d, p, cells, solves):
    import torch
    mesh = W.structured_mesh(d, cells, p)
    field = W.fourier_perturbed_field(2, 0.2, 5) if d == 2 else W.taylor_green_field(0.2)
    st = W.make_state(mesh, field, 7, noise=0.01)
    lm = lib_mesh(W.Workload("repeat", mesh, st, dict(gamma=1.4, Pr=0.72, Re=1e3, Minf=0.2, alpha=W.dirk_alpha())))
    K, R = lm.assemble_condensed(dev(st.u), dev(st.q), dev(st.uhat))
    first, its, rr = lm.trace_solve(K, R, rtol=1e-12, max_iter=2000)
    first = first.clone()
    assert rr <= 1e-12
    for k in range(solves):
        dU, n, r = lm.trace_solve(K, R, rtol=1e-12, max_iter=2000)
        assert n == its and r == rr and torch.equal(dU, first), k
