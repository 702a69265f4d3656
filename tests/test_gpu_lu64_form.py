"""The schedule chooses the FP64 LU's form at every element size: 0 = DFMA updates, 1 =
digit products on the tensor cores; the default is the digit form from 64 u-unknowns."""
import numpy as np
import pytest

from paper_1605_01020_gb300 import workloads as W
from gpu_helpers import dev, host, lib_mesh, rel_err

pytestmark = pytest.mark.gpu


def _assemble(lm, st):
    K, R = lm.assemble_condensed(dev(st.u), dev(st.q), dev(st.uhat))
    assert (lm.element_status() == 0).all()
    return host(K), host(R)


@pytest.mark.parametrize("d,p,default", [(2, 2, 0), (2, 3, 1), (3, 2, 1)])       # 36, 64, 135 u-unknowns
def test_the_form_is_the_callers_choice(d, p, default):
    mesh = W.structured_mesh(d, 2, p)
    field = W.fourier_perturbed_field(2, 0.2, 5, amp=0.05) if d == 2 else W.taylor_green_field(0.2)
    st = W.make_state(mesh, field, 7, noise=0.01)
    lm = lib_mesh(W.Workload("form", mesh, st, dict(gamma=1.4, Pr=0.72, Re=1e3, Minf=0.2, alpha=W.dirk_alpha())))
    assert lm.get_schedule()["lu_tensor"] == default
    usual = _assemble(lm, st)
    out = []
    for form in (0, 1):
        lm.set_schedule(lu_tensor=form)
        out.append(_assemble(lm, st))
    assert all(np.array_equal(a, b) for a, b in zip(out[default], usual))
    # the two forms round differently (equal bits: one kernel ran for both values) and agree
    assert not np.array_equal(out[0][0], out[1][0])
    assert rel_err(out[1][0], out[0][0]) <= 1e-11
    lm.set_schedule(lu_tensor=0, lu_panel=32)
    assert rel_err(_assemble(lm, st)[0], out[0][0]) <= 1e-11


def test_mixed_orders_default():
    from paper_1605_01020_gb300 import iedg
    for orders, want in (([1, 2, 1, 2, 2, 1, 2, 1], 1), ([1] * 8, 0)):
        mm = W.structured_mesh_mixed(3, (2, 2, 2), np.array(orders))
        lm = iedg.MixedOrderMesh(mm.node_xyz, mm.elem_trace, mm.n_trace, mm.orders, mm.face_degree, gamma=1.4, Pr=0.72,
                                 Re=1e3, Minf=0.2, alpha=W.dirk_alpha())
        assert lm.get_schedule()["lu_tensor"] == want
