"""The FP64 LU's digit form on element systems whose rows and columns span a wide range (low
Reynolds and Mach numbers, flat cells).  The rounding errors of an FP64 elimination are
measured on the oracle's element systems against extended precision: largest entry of K,
worst of the 25 component blocks, median entry.  On the GPU both forms start from the same
element matrices, so their difference is the sum of two such errors, about 1.5 times one of
them; 4 times is allowed for the scatter of maxima.  (Without the scaling of the panel's
unknowns, level 8 of the products and the rounding of the operands the ratios were 7 to 20
on the medians of the wide systems, and up to 300.)"""
import numpy as np
import pytest

from paper_1605_01020_gb300 import workloads as W
from gpu_helpers import dev, host, lib_mesh
from oracle_helpers import problem
from oracle import iedg as oiedg

pytestmark = pytest.mark.gpu


def _condense(At, Bt, Ct, Dt, dtype):
    """Dt - Ct At^-1 Bt by elimination with partial pivoting in the given precision."""
    nu = len(At)
    A = np.block([[At, Bt], [Ct, Dt]]).astype(dtype)
    for j in range(nu):
        p = j + int(np.argmax(np.abs(A[j:nu, j])))
        if p != j:
            A[[j, p]] = A[[p, j]]
        A[j + 1:, j + 1:] -= np.outer(A[j + 1:, j] / A[j, j], A[j, j + 1:])
    return A[nu:, nu:]


def _errors(K, ref):
    E, m = np.abs(K - ref), K.shape[-1]
    blocks = [E[:, i, k].max() / np.abs(ref[:, i, k]).max() for i in range(m) for k in range(m)
              if np.abs(ref[:, i, k]).max() > 0]
    nz = ref != 0
    return np.array([E.max() / np.abs(ref).max(), max(blocks), np.median(E[nz] / np.abs(ref[nz]))], dtype=float)


@pytest.mark.parametrize("Re,M,ratio", [(2.5e5, 0.2, 1.0), (1.0, 0.02, 50.0), (1.0, 0.01, 1e4), (1e-3, 1e-4, 100.0),
                                        (1e-3, 1e-4, 1000.0)])
def test_digit_form_differs_by_rounding_errors(Re, M, ratio):
    mesh = W.structured_mesh(3, 2, 2)
    st = W.make_state(mesh, W.taylor_green_field(M), 7, noise=0.01)
    mesh.node_xyz = mesh.node_xyz.copy()
    mesh.node_xyz[..., 1] /= ratio
    st.q = st.q.copy()
    st.q[..., 1] *= ratio
    wl = W.Workload("wide", mesh, st, dict(gamma=1.4, Pr=0.72, Re=Re, Minf=M, alpha=W.dirk_alpha()))
    pb = problem(mesh, wl.params)
    Nb = mesh.elem_trace.shape[1]
    row_ptr, col = oiedg.bsr_pattern(mesh.elem_trace, mesh.n_trace)
    K = {t: np.zeros((len(col), 5, 5), dtype=t) for t in (np.float64, np.longdouble)}
    for e in range(mesh.n_elem):
        system = pb.qelim(pb.element_blocks(e, st.u, st.q, st.uhat))[:4]
        tr = mesh.elem_trace[e]
        pos = np.array([[oiedg.bsr_find(row_ptr, col, r, c) for c in tr] for r in tr]).reshape(-1)
        for t in K:
            Ke = _condense(*system, t).reshape(5, Nb, 5, Nb).transpose(1, 3, 0, 2)
            np.add.at(K[t], pos, Ke.reshape(-1, 5, 5))
    fp64 = _errors(K[np.float64], K[np.longdouble])
    lm = lib_mesh(wl)
    out = []
    for form in (0, 1):
        lm.set_schedule(lu_tensor=form)
        out.append(host(lm.assemble_condensed(dev(st.u), dev(st.q), dev(st.uhat))[0]))
        assert (lm.element_status() == 0).all()
    diff = _errors(out[1], out[0])
    print(f"Re {Re} M {M} ratio {ratio}: FP64 elimination {fp64}, digits - DFMA {diff}")
    assert (diff <= 4 * fp64).all(), (diff, fp64)
