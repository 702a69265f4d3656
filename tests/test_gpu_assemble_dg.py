"""FP64 element matrices from digit products on the tensor cores: column tiles that straddle
pairs and end short (degrees 2..4, two elements of unlike shape), and operands whose
scales differ widely (a mesh of size 1e-3 and of size 1e3 against a unit state: lifting
operators, point coefficients and mass terms move by powers of the size).  Against the
oracle at the tolerance of the other FP64 parity tests."""
import numpy as np
import pytest

from oracle import iedg as oiedg
from paper_1605_01020_gb300 import workloads as W
from gpu_helpers import bsr_row_err, dev, host, lib_mesh, rel_err
from oracle_helpers import problem

pytestmark = pytest.mark.gpu
TOL = 1e-11


@pytest.mark.parametrize("p,size,stab", [(2, 1.0, 1), (2, 1e-3, 0), (3, 1e3, 0), (3, 1e-3, 1)])
def test_digit_assembly_parity(p, size, stab):
    mesh = W.structured_mesh(3, (2, 2, 2), p, mapping=W.stretched_mapping(3, ratio=3.0))
    st = W.make_state(mesh, W.taylor_green_field(0.2), 7, noise=0.01, uref_shift=0.01)
    mesh.node_xyz = mesh.node_xyz * size
    st.q = st.q / size
    # Re and the stage coefficient follow the size, so that the terms keep their balance
    wl = W.Workload("dg", mesh, st, dict(gamma=1.4, Pr=0.72, Re=1e3 / size, Minf=0.2, alpha=W.dirk_alpha() / size,
                                         stab=stab))
    pb = problem(mesh, wl.params)
    Ke, Re = zip(*[pb.condense_qelim(e, st.u, st.q, st.uhat, st.u_ref) for e in range(mesh.n_elem)])
    row_ptr, _, vals, R = oiedg.assemble(mesh.elem_trace, mesh.n_trace, np.array(Ke), np.array(Re))
    lm = lib_mesh(wl)
    K_d, R_d = lm.assemble_condensed(dev(st.u), dev(st.q), dev(st.uhat), u_ref=dev(st.u_ref))
    assert (lm.element_status() == 0).all()
    assert bsr_row_err(row_ptr, host(K_d), vals, range(mesh.n_trace)) <= TOL
    assert rel_err(host(R_d), R, floor=np.abs(np.array(Re)).max()) <= TOL
    du_d, dq_d = lm.back_substitute(dev(st.duhat))
    upd = [pb.back_substitute_qelim(e, st.u, st.q, st.uhat, st.duhat, st.u_ref) for e in range(mesh.n_elem)]
    assert rel_err(host(du_d), np.array([x[0] for x in upd])) <= TOL


def test_nonfinite_operand_is_flagged():
    """A NaN in one element's state reaches only that element's blocks and status."""
    from paper_1605_01020_gb300 import iedg
    mesh = W.structured_mesh(3, (2, 2, 2), 2)
    st = W.make_state(mesh, W.taylor_green_field(0.2), 7, noise=0.01)
    u = st.u.copy()
    u[3, 13, 1] = np.nan                      # the interior node: volume points only
    wl = W.Workload("nan", mesh, st, dict(gamma=1.4, Pr=0.72, Re=1e3, Minf=0.2, alpha=W.dirk_alpha()))
    lm = lib_mesh(wl)
    lm.assemble_condensed(dev(u), dev(st.q), dev(st.uhat))
    s = lm.element_status()
    assert s[3] == iedg.ELEM_NONFINITE and (np.delete(s, 3) == iedg.ELEM_OK).all(), s
