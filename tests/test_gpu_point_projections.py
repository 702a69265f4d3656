"""Residual projections in 3D, one direction at a time, against the oracle's dense ones:
degrees 1..4 with the smallest and the largest quadrature rule a handle takes, curved
elements, with and without the time term.  Same tolerance as the other FP64 outputs."""
import numpy as np
import pytest

from paper_1605_01020_gb300 import iedg, workloads as W
from gpu_helpers import dev, host, rel_err
from oracle_helpers import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,extra,ref", [(1, 1, True), (1, 3, False), (2, 1, False), (2, 3, True), (3, 3, True),
                                         (4, 1, True), (4, 3, False)])
def test_residual_with_other_quadrature_rules(p, extra, ref):
    mesh = W.structured_mesh(3, 2, p, mapping=W.stretched_mapping(5, ratio=3.0))
    st = W.make_state(mesh, W.taylor_green_field(0.2), 3, noise=0.01, uref_shift=0.01)
    prm = dict(gamma=1.4, Pr=0.72, Re=200.0, Minf=0.2, alpha=W.dirk_alpha())
    uref = st.u_ref if ref else None
    _, Ru, Rh, Rfl = problem(mesh, prm, quad_extra=extra).residual(st.u, st.q, st.uhat, uref)
    h = iedg.Mesh(mesh.node_xyz, mesh.elem_trace, mesh.n_trace, p, quad_extra=extra, **prm)
    out = h.eval_residual(dev(st.u), dev(st.uhat), q=dev(st.q), u_ref=dev(uref))
    assert rel_err(host(out["r_u"]), Ru) <= 1e-11
    assert rel_err(host(out["r_fl"]), Rfl, floor=np.abs(Rh).max()) <= 1e-11
