"""The digit assembly's waits give up in order: with no poll allowed its blocks leave NaN
instead of waiting for one another, which a DFMA LU reports as IEDG_ELEM_NONFINITE, on uniform
and mixed-order meshes, and the next call with the usual limit gives the usual results."""
import numpy as np
import pytest

from paper_1605_01020_gb300 import workloads as W
from gpu_helpers import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,cells", [(2, (3, 2, 2)), (3, (7, 6, 5)), (4, (2, 2, 2))])
def test_waits_give_up_and_recover(p, cells):
    from paper_1605_01020_gb300 import iedg
    mesh = W.structured_mesh(3, cells, p)
    st = W.make_state(mesh, W.taylor_green_field(0.2), 7, noise=0.01)
    wl = W.Workload("waits", mesh, st, dict(gamma=1.4, Pr=0.72, Re=1e3, Minf=0.2, alpha=W.dirk_alpha()))
    lm = iedg.mesh_from_workload(wl)
    lm.set_schedule(lu_tensor=0)

    def run():
        K, R = lm.assemble_condensed(dev(st.u), dev(st.q), dev(st.uhat))
        return host(K), host(R), lm.element_status()

    K0, R0, status = run()
    assert (status == iedg.ELEM_OK).all(), status
    lm.set_fault_injection(tc_wait_limit=-1)
    _, _, status = run()
    assert (status == iedg.ELEM_NONFINITE).all(), status
    lm.set_fault_injection()
    K1, R1, status = run()
    assert (status == iedg.ELEM_OK).all(), status
    assert np.array_equal(K1, K0) and np.array_equal(R1, R0)


def test_mixed_orders():
    from paper_1605_01020_gb300 import iedg
    orders = np.array([2, 3, 4, 3, 2, 3, 4, 2])
    mm = W.structured_mesh_mixed(3, (2, 2, 2), orders)
    lm = iedg.MixedOrderMesh(mm.node_xyz, mm.elem_trace, mm.n_trace, mm.orders, mm.face_degree, gamma=1.4, Pr=0.72,
                             Re=1e3, Minf=0.2, alpha=W.dirk_alpha())
    lm.set_schedule(lu_tensor=0)
    field = W.taylor_green_field(0.2)
    u = dev(np.concatenate([field(x) for x in mm.node_xyz]))
    q = dev(np.zeros(lm._qshape))
    uhat = dev(np.tile(field(np.zeros((1, 3))), (mm.n_trace, 1)))
    K0, _ = lm.assemble_condensed(u, q, uhat)
    K0 = host(K0)
    assert (lm.element_status() == iedg.ELEM_OK).all()
    lm.set_fault_injection(tc_wait_limit=-1)
    lm.assemble_condensed(u, q, uhat)
    assert (lm.element_status() == iedg.ELEM_NONFINITE).all(), lm.element_status()
    lm.set_fault_injection()
    K1, _ = lm.assemble_condensed(u, q, uhat)
    assert (lm.element_status() == iedg.ELEM_OK).all() and np.array_equal(host(K1), K0)
