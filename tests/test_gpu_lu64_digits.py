"""FP64 partial LU with digit-split tensor-core updates (lu_tensor = 1) at the element
sizes where its tiles are ragged: fewer u-unknowns than a panel, a last panel of a few
columns, rows and columns below one tile.  Against the oracle, at the tolerance of the
other FP64 parity tests."""
import numpy as np
import pytest

from oracle import iedg as oiedg
from paper_1605_01020_gb300 import workloads as W
from gpu_helpers import bsr_row_err, dev, host, lib_mesh, rel_err
from oracle_helpers import problem

pytestmark = pytest.mark.gpu
TOL = 1e-11


@pytest.mark.parametrize("d,p", [(2, 1), (2, 2), (3, 1), (3, 2)])   # n x nu: 32 x 16, 68 x 36, 80 x 40, 265 x 135
def test_digit_lu_ragged_tiles(d, p):
    mesh = W.structured_mesh(d, 2, p, mapping=W.stretched_mapping(3, ratio=3.0))
    field = W.fourier_perturbed_field(2, 0.2, 5, amp=0.05) if d == 2 else W.taylor_green_field(0.2)
    st = W.make_state(mesh, field, 7, noise=0.01, uref_shift=0.01)
    wl = W.Workload("ragged", mesh, st, dict(gamma=1.4, Pr=0.72, Re=1e3, Minf=0.2, alpha=W.dirk_alpha()))
    pb = problem(mesh, wl.params)
    Ke, Re = zip(*[pb.condense_qelim(e, st.u, st.q, st.uhat, st.u_ref) for e in range(mesh.n_elem)])
    row_ptr, _, vals, R = oiedg.assemble(mesh.elem_trace, mesh.n_trace, np.array(Ke), np.array(Re))
    lm = lib_mesh(wl)
    lm.set_schedule(lu_tensor=1)
    K_d, R_d = lm.assemble_condensed(dev(st.u), dev(st.q), dev(st.uhat), u_ref=dev(st.u_ref))
    assert (lm.element_status() == 0).all()
    assert bsr_row_err(row_ptr, host(K_d), vals, range(mesh.n_trace)) <= TOL
    assert rel_err(host(R_d), R, floor=np.abs(np.array(Re)).max()) <= TOL
    du_d, dq_d = lm.back_substitute(dev(st.duhat))
    upd = [pb.back_substitute_qelim(e, st.u, st.q, st.uhat, st.duhat, st.u_ref) for e in range(mesh.n_elem)]
    assert rel_err(host(du_d), np.array([x[0] for x in upd])) <= TOL
    assert rel_err(host(dq_d), np.array([x[1] for x in upd])) <= TOL
