"""The digit assembly's waits give up in order: with no poll allowed its blocks leave NaN
(IEDG_ELEM_NONFINITE) instead of waiting for one another, on the FP64 form of uniform and
mixed-order meshes and in the FP64 fallback of the mixed forms, and the next call with the
usual limit gives the usual results."""
import numpy as np
import pytest

from paper_1605_01020_gb300 import workloads as W
from gpu_helpers import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,cells,precision", [(2, (3, 2, 2), 0), (3, (7, 6, 5), 0), (4, (2, 2, 2), 0), (3, (2, 2, 2), 1)])
def test_waits_give_up_and_recover(p, cells, precision):
    from paper_1605_01020_gb300 import iedg
    mesh = W.structured_mesh(3, cells, p)
    st = W.make_state(mesh, W.taylor_green_field(0.2), 7, noise=0.01)
    wl = W.Workload("waits", mesh, st, dict(gamma=1.4, Pr=0.72, Re=1e3, Minf=0.2, alpha=W.dirk_alpha()))
    lm = iedg.mesh_from_workload(wl, precision=precision)
    fall = dict(refine_iters=0) if precision else {}
    usual = iedg.ELEM_FALLBACK if precision else iedg.ELEM_OK

    def run():
        K, R = lm.assemble_condensed(dev(st.u), dev(st.q), dev(st.uhat))
        return host(K), host(R), lm.element_status()

    lm.set_fault_injection(**fall)
    K0, R0, status = run()
    assert (status == usual).all(), status
    lm.set_fault_injection(asm_wait_limit=-1, **fall)
    _, _, status = run()
    assert (status == iedg.ELEM_NONFINITE).all(), status
    lm.set_fault_injection(**fall)
    K1, R1, status = run()
    assert (status == usual).all(), status
    assert np.array_equal(K1, K0) and np.array_equal(R1, R0)


def test_mixed_orders():
    from paper_1605_01020_gb300 import iedg
    orders = np.array([2, 3, 4, 3, 2, 3, 4, 2])
    mm = W.structured_mesh_mixed(3, (2, 2, 2), orders)
    lm = iedg.MixedOrderMesh(mm.node_xyz, mm.elem_trace, mm.n_trace, mm.orders, mm.face_degree, gamma=1.4, Pr=0.72,
                             Re=1e3, Minf=0.2, alpha=W.dirk_alpha())
    field = W.taylor_green_field(0.2)
    u = dev(np.concatenate([field(x) for x in mm.node_xyz]))
    q = dev(np.zeros(lm._qshape))
    uhat = dev(np.tile(field(np.zeros((1, 3))), (mm.n_trace, 1)))
    K0, _ = lm.assemble_condensed(u, q, uhat)
    K0 = host(K0)
    assert (lm.element_status() == iedg.ELEM_OK).all()
    lm.set_fault_injection(asm_wait_limit=-1)
    lm.assemble_condensed(u, q, uhat)
    assert (lm.element_status() == iedg.ELEM_NONFINITE).all(), lm.element_status()
    lm.set_fault_injection()
    K1, _ = lm.assemble_condensed(u, q, uhat)
    assert (lm.element_status() == iedg.ELEM_OK).all() and np.array_equal(host(K1), K0)
