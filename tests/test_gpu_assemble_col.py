"""Assembly of small elements with a thread per column (2D of degree 1..3, 3D of degree
1), FP64 and FP32, both stabilisations, on curved meshes whose columns do not fill the
last CTA.  K and R against the oracle at the tolerances of the other parity tests."""
import numpy as np
import pytest

from oracle import iedg as oiedg
from paper_1605_01020_gb300 import iedg, workloads as W
from gpu_helpers import bsr_row_err, dev, host, rel_err
from oracle_helpers import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("d,p,stab", [(2, 1, 1), (2, 2, 0), (2, 3, 1), (3, 1, 0), (3, 1, 1)])
def test_column_assembly_parity(d, p, stab, precision):
    mesh = W.structured_mesh(d, (3, 2, 2)[:d], p, mapping=W.stretched_mapping(3, ratio=3.0))
    field = W.fourier_perturbed_field(2, 0.2, 5, amp=0.05) if d == 2 else W.taylor_green_field(0.2)
    st = W.make_state(mesh, field, 7, noise=0.01, uref_shift=0.01)
    wl = W.Workload("col", mesh, st, dict(gamma=1.4, Pr=0.72, Re=1e3, Minf=0.2, alpha=W.dirk_alpha(), stab=stab))
    pb = problem(mesh, wl.params)
    Ke, Re = zip(*[pb.condense_qelim(e, st.u, st.q, st.uhat, st.u_ref) for e in range(mesh.n_elem)])
    row_ptr, _, vals, R = oiedg.assemble(mesh.elem_trace, mesh.n_trace, np.array(Ke), np.array(Re))
    lm = iedg.mesh_from_workload(wl, precision=precision)
    K_d, R_d = lm.assemble_condensed(dev(st.u), dev(st.q), dev(st.uhat), u_ref=dev(st.u_ref))
    assert (lm.element_status() == 0).all()
    assert bsr_row_err(row_ptr, host(K_d), vals, range(mesh.n_trace)) <= (1e-11 if precision == 0 else 1e-4)
    assert rel_err(host(R_d), R, floor=np.abs(np.array(Re)).max()) <= (1e-11 if precision == 0 else 1e-10)
