"""FP32 partial LU at the element sizes where its tiles are ragged: fewer u-unknowns than a
panel, a last panel whose columns are not on 16-byte boundaries (135 = 4 x 32 + 7), fewer
trailing columns than a tile; FFMA and deferred
tensor-core forms.  K against the FP64 path to FP32 accuracy, R and the updates to the
refinement's."""
import numpy as np
import pytest

from paper_1605_01020_gb300 import iedg, workloads as W
from gpu_helpers import dev, host, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lu_tensor", [0, 1])
@pytest.mark.parametrize("d,p", [(2, 1), (2, 2), (3, 1), (3, 2)])     # n x nu: 32 x 16, 68 x 36, 80 x 40, 265 x 135
def test_fp32_lu_ragged_tiles(d, p, lu_tensor):
    mesh = W.structured_mesh(d, 2, p, mapping=W.stretched_mapping(3, ratio=3.0))
    field = W.fourier_perturbed_field(2, 0.2, 5, amp=0.05) if d == 2 else W.taylor_green_field(0.2)
    st = W.make_state(mesh, field, 7, noise=0.01, uref_shift=0.01)
    prm = dict(gamma=1.4, Pr=0.72, Re=1e3, Minf=0.2, alpha=W.dirk_alpha())
    args = [dev(st.u), dev(st.q), dev(st.uhat)]
    out = []
    for precision in (0, 1):
        m = iedg.Mesh(mesh.node_xyz, mesh.elem_trace, mesh.n_trace, p, precision=precision, **prm)
        if precision:
            m.set_schedule(lu_tensor=lu_tensor)
        K, R = m.assemble_condensed(*args, u_ref=dev(st.u_ref))
        assert (m.element_status() == 0).all()
        out.append([host(t) for t in (K, R, *m.back_substitute(dev(st.duhat)))])
    assert rel_err(out[1][0], out[0][0]) <= 1e-4
    for a, b in zip(out[1][1:], out[0][1:]):
        assert rel_err(a, b) <= 1e-10
