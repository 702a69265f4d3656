"""The FP64 digit assembly is as accurate as FP64 sums: K of the default path (digit assembly
and LU) against the oracle's element systems condensed in extended precision, compared with
an FP64 elimination of the same systems.  Both sides' assembly and elimination contribute
errors of that size and the device's coefficients differ from the oracle's by rounding: a
factor 3 is allowed.  (With columns scaled by a bound from the factors' separate maxima,
6 bits too high on most, the median entry was at 3.8 times.)"""
import numpy as np
import pytest
import scipy.linalg

from oracle import iedg as oiedg
from paper_1605_01020_gb300 import workloads as W
from gpu_helpers import dev, host, lib_mesh
from oracle_helpers import problem

pytestmark = pytest.mark.gpu


def _slices(A, axis):
    """A as three float64 parts of 20 bits below the largest entry along `axis`, so that
    products of parts are exact over a thousand terms."""
    out, rest = [], np.array(A)
    top = np.abs(A).max(axis, keepdims=True)
    unit = np.ldexp(1.0, np.frexp(np.where(top > 0, top, 1.0))[1])
    for _ in range(3):
        unit = unit * 2.0 ** -20
        out.append(np.rint(rest / unit) * unit)
        rest = rest - out[-1]
    return out


def _product(As, B):
    """A B in extended precision, A given by its row slices, B = (high, low) parts."""
    parts = [a @ b for b in _slices(B[0], 0) for a in As] + [sum(As) @ B[1]]
    return sum((p.astype(np.longdouble) for p in sorted(parts, key=lambda p: np.abs(p).max())), np.longdouble(0))


def _condense_extended(At, Bt, Ct, Dt):
    """Dt - Ct At^-1 Bt with the solution refined to twice FP64's length."""
    lu, As, Cs = scipy.linalg.lu_factor(At), _slices(At, 1), _slices(Ct, 1)
    hi, lo = scipy.linalg.lu_solve(lu, Bt), np.zeros_like(Bt)
    for _ in range(4):
        r = (Bt.astype(np.longdouble) - _product(As, (hi, lo))).astype(np.float64)
        x = hi.astype(np.longdouble) + lo + scipy.linalg.lu_solve(lu, r)
        hi = x.astype(np.float64)
        lo = (x - hi).astype(np.float64)
    return Dt.astype(np.longdouble) - _product(Cs, (hi, lo))


def _condense(At, Bt, Ct, Dt):
    """The same by plain FP64 elimination with partial pivoting."""
    nu = len(At)
    A = np.block([[At, Bt], [Ct, Dt]])
    for j in range(nu):
        p = j + int(np.argmax(np.abs(A[j:nu, j])))
        A[[j, p]] = A[[p, j]]
        A[j + 1:, j + 1:] -= np.outer(A[j + 1:, j] / A[j, j], A[j, j + 1:])
    return A[nu:, nu:]


@pytest.mark.parametrize("Re,M,ratio", [(1e5, 0.1, 1000.0)])
def test_condensed_entries(Re, M, ratio):
    p = 3
    mesh = W.structured_mesh(3, 2, p)
    st = W.make_state(mesh, W.taylor_green_field(M), 7, noise=0.01)
    mesh.node_xyz = mesh.node_xyz.copy()
    mesh.node_xyz[..., 1] /= ratio
    st.q = st.q.copy()
    st.q[..., 1] *= ratio
    wl = W.Workload("flat", mesh, st, dict(gamma=1.4, Pr=0.72, Re=Re, Minf=M, alpha=W.dirk_alpha()))
    pb = problem(mesh, wl.params)
    Nb = mesh.elem_trace.shape[1]
    row_ptr, col = oiedg.bsr_pattern(mesh.elem_trace, mesh.n_trace)
    K = {f: np.zeros((len(col), 5, 5), dtype=t) for f, t in ((_condense, np.float64), (_condense_extended, np.longdouble))}
    for e in range(mesh.n_elem):
        system = pb.qelim(pb.element_blocks(e, st.u, st.q, st.uhat))[:4]
        tr = mesh.elem_trace[e]
        pos = np.array([[oiedg.bsr_find(row_ptr, col, r, c) for c in tr] for r in tr]).reshape(-1)
        for f in K:
            np.add.at(K[f], pos, f(*system).reshape(5, Nb, 5, Nb).transpose(1, 3, 0, 2).reshape(-1, 5, 5))
    ref = K[_condense_extended]
    nz = ref != 0

    def err(x):
        d = np.abs(x - ref)
        blocks = [d[:, i, k].max() / np.abs(ref[:, i, k]).max() for i in range(5) for k in range(5)]
        return np.array([d.max() / np.abs(ref).max(), max(blocks), np.median((d[nz] / np.abs(ref[nz])).astype(float))], dtype=float)

    lm = lib_mesh(wl)
    K_d, _ = lm.assemble_condensed(dev(st.u), dev(st.q), dev(st.uhat))
    assert (lm.element_status() == 0).all()
    got, fp64 = err(host(K_d)), err(K[_condense])
    print(f"Re {Re} M {M} ratio {ratio}: FP64 elimination {fp64}, device {got}")
    assert (got <= 3 * fp64).all(), (got, fp64)
