"""FP32 hexahedra assembled with two threads per column (uniform meshes) against the
assembly of meshes with mixed orders given the same elements: the same FP32 operations in
the same order, so the factored systems may differ only where the compiler contracts a
product differently.  Degrees 2..4 (two, two and three z layers a thread), both
stabilisations, curved elements."""
import numpy as np
import pytest

from paper_1605_01020_gb300 import iedg, workloads as W
from gpu_helpers import dev, host, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,stab", [(2, 0), (2, 1), (3, 0), (3, 1), (4, 1)])
def test_uniform_and_mixed_order_assembly_agree(p, stab):
    mesh = W.structured_mesh(3, (3, 2, 2), p, mapping=W.stretched_mapping(3, ratio=3.0))
    st = W.make_state(mesh, W.taylor_green_field(0.2), 7, noise=0.01, uref_shift=0.01)
    prm = dict(gamma=1.4, Pr=0.72, Re=1e3, Minf=0.2, alpha=W.dirk_alpha())
    a = iedg.Mesh(mesh.node_xyz, mesh.elem_trace, mesh.n_trace, p, precision=1, stab=stab, **prm)
    E = mesh.n_elem
    b = iedg.MixedOrderMesh(list(mesh.node_xyz), list(mesh.elem_trace), mesh.n_trace, np.full(E, p),
                            np.zeros((E, 6), dtype=int), precision=1, stab=stab, **prm)
    b.set_schedule(lu_tensor=0)              # the uniform handle's LU form
    flat = lambda x: dev(x.reshape(-1, *x.shape[2:]))
    Ka, Ra = a.assemble_condensed(dev(st.u), dev(st.q), dev(st.uhat), u_ref=dev(st.u_ref))
    Kb, Rb = b.assemble_condensed(flat(st.u), flat(st.q), dev(st.uhat), u_ref=flat(st.u_ref))
    assert (a.element_status() == 0).all() and (b.element_status() == 0).all()
    assert rel_err(host(Ka), host(Kb)) <= 1e-5 and rel_err(host(Ra), host(Rb)) <= 1e-11
