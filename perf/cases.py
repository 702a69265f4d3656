"""The work a user of this library has it do, case by case.

A case is one call sequence of a flow solver on one mesh handle, through the binding in
paper_1605_01020_gb300/iedg.py:
  residual   iedg_eval_residual with the gradient lifted from (u, uhat): what the time
             stepper evaluates for its initial guesses and stopping tests;
  newton     residual at a given (u, q, uhat), condensed linearisation, back-substitution
             of a trace increment: the element-local part of one Newton step;
  iteration  the same with the library's own trace solve in the middle: a whole Newton step;
  trace      the GMRES solve of the condensed system alone.
Meshes are periodic blocks of curved or plain hexahedra or quadrilaterals, and blocks of
mixed orders, with or without far-field and wall faces.  The state is a smooth field with
seeded phases and 1 % nodal noise; the stage reference state differs from it by 1 %.

`exact` evaluates the same discretisation with plain torch in 64 bits: pointwise
Jacobians by torch.func, dense element systems, torch.linalg.solve.
"""
import itertools
import math

import numpy as np
import torch

from paper_1605_01020_gb300 import iedg, workloads

F64 = torch.float64
ALPHA = workloads.dirk_alpha()
PREC = {"fp64": 0, "fp32": 1, "tf32": 2, "bf16": 3}
RTOL = 1e-12                       # the time stepper's tolerance of the trace solve


# ----------------------------------------------------------------------------- cases
def _case(name, op, d, cells, p, prec="fp64", stab="lf", shape="plain", scale=False, precond="jacobi"):
    """cells "16x16x16"; p one digit, or the digits of the orders that are mixed;
    shape: plain | curved | wall (mixed orders only)."""
    c = {"op": op, "d": d, "cells": cells, "p": p, "prec": prec, "stab": stab, "shape": shape, "scale": scale,
         "precond": precond}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: the stopping test of a 2D run
        _case("residual_2d_p2", "residual", 2, "8x8", "2"),
        # a whole Newton step of the same run: launches and the trace solve's latency count
        _case("iteration_2d_p2", "iteration", 2, "8x8", "2"),
        # an ordinary 2D run with Roe's flux on a stretched, sheared mesh of odd size
        _case("newton_2d_p3_roe", "newton", 2, "37x23", "3", stab="roe", shape="curved"),
        # the paper's degree k = 2 in 3D, full FP64
        _case("newton_3d_p2", "newton", 3, "14x13x11", "2"),
        # the headline workload: 3D p = 3, 16^3, FP64 and with FP32 factors and FP64 refinement
        _case("newton_3d_p3", "newton", 3, "16x16x16", "3"),
        _case("newton_3d_p3_fp32", "newton", 3, "16x16x16", "3", prec="fp32"),
        # the highest degree on a stretched, sheared mesh that does not fill the chip evenly
        _case("newton_3d_p4", "newton", 3, "7x6x5", "4", shape="curved"),
        _case("newton_3d_p4_fp32", "newton", 3, "7x6x5", "4", prec="fp32", stab="roe", shape="curved"),
        # rounded Schur operands with the element systems scaled by their mass matrices
        _case("newton_3d_p3_tf32", "newton", 3, "9x8x7", "3", prec="tf32", scale=True),
        # orders 2, 3, 4 side by side; the second with walls and far-field faces
        _case("newton_orders", "newton", 3, "6x6x9", "234"),
        _case("newton_orders_fp32_wall", "newton", 3, "5x5x7", "234", prec="fp32", shape="wall"),
        # the condensed system's solve for the time stepper's tolerance
        _case("trace_3d_p3", "trace", 3, "6x6x6", "3"),
    ]


def _cells(c):
    return [int(x) for x in c["cells"].split("x")]


def draw(rng):
    def cells(d, lo, hi):
        n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        out = []
        for r in range(d):
            k = max(2, round((n ** (1.0 / (d - r))) * rng.uniform(0.8, 1.25)) if r < d - 1 else round(n))
            out.append(k)
            n = max(n / k, 2.0)
        return "x".join(str(k) for k in out)

    kind = rng.choice(["newton", "newton", "newton", "newton", "residual", "iteration", "trace", "orders", "orders"])
    stab, shape = rng.choice(["lf", "lf", "roe"]), rng.choice(["plain", "curved"])
    if kind == "orders":
        prec = rng.choice(["fp64", "fp32"])
        return _case(None, "newton", 3, cells(3, 16, 256), rng.choice(["234", "23", "34"]), prec, stab,
                     rng.choice(["plain", "wall"]))
    if kind == "trace":
        d = rng.choice([2, 3])
        return _case(None, "trace", d, cells(d, 16, 200), str(rng.randint(1, 3)), "fp64", stab, shape,
                     precond=rng.choice(["jacobi", "jacobi", "jacobi", "bilu0"]))
    if kind in ("residual", "iteration"):
        d = rng.choice([2, 3])
        return _case(None, kind, d, cells(d, 16, 256), str(rng.randint(1, 3)), "fp64", stab, shape)
    d = rng.choice([2, 3, 3, 3])
    if d == 2:
        return _case(None, "newton", 2, cells(2, 30, 1500), str(rng.randint(1, 3)), rng.choice(["fp64", "fp32"]), stab,
                     shape)
    p = rng.randint(1, 4)
    prec = rng.choice(["fp64", "fp64", "fp32", "fp32", "tf32", "bf16"])
    scale = prec != "fp64" and rng.random() < 0.3
    return _case(None, "newton", 3, cells(3, 16, [4096, 4096, 2000, 300][p - 1]), str(p), prec, stab, shape, scale)


# ---------------------------------------------------------------------------- meshes
def _multi(n, d):
    """[n^d, d] multi-indices, first direction fastest."""
    return np.array([t[::-1] for t in itertools.product(range(n), repeat=d)], dtype=np.int64).reshape(-1, d)


def _mapping(X):
    """Smooth periodic map: y graded towards one plane (cell sizes 1 : 4), x and z sheared."""
    beta, Y = 0.6, X.copy()
    xi, eta = X[..., 0], X[..., 1]
    Y[..., 1] = eta - beta / (2 * np.pi) * np.sin(2 * np.pi * eta)
    Y[..., 0] = xi + 0.2 / (2 * np.pi) * np.sin(2 * np.pi * eta + 0.7)
    if X.shape[-1] == 3:
        Y[..., 2] = X[..., 2] + 0.2 / (2 * np.pi) * np.sin(2 * np.pi * xi + 1.9)
    return Y


class _Mesh:
    """Per-element lists X (nodes), trace (slot -> trace node); uniform meshes also as arrays."""

    def __init__(self, c):
        d, N = c["d"], _cells(c)
        self.d, self.m, self.mixed = d, d + 2, len(c["p"]) > 1
        if self.mixed:
            rng = np.random.default_rng(sum(N))
            levels = [int(x) for x in c["p"]]
            orders = rng.choice(np.array(levels), size=int(np.prod(N)),
                                p={3: [0.3, 0.5, 0.2], 2: [0.5, 0.5]}[len(levels)])
            mm = workloads.structured_mesh_mixed(d, N, orders, boundary=(1, 2, 0) if c["shape"] == "wall" else None)
            self.orders, self.face_degree, self.face_kind = mm.orders, mm.face_degree, mm.face_kind
            self.X, self.trace, self.T = mm.node_xyz, mm.elem_trace, mm.n_trace
        else:
            p = int(c["p"])
            nodes, E = _multi(p + 1, d), int(np.prod(N))
            cell = np.stack(np.unravel_index(np.arange(E), N[::-1])[::-1], -1)
            xi = 0.5 * (1.0 + workloads.gll_positions(p))
            X = (cell[:, None, :] + xi[nodes][None]) / np.array(N, dtype=np.float64)
            self.X = _mapping(X) if c["shape"] == "curved" else X
            self.bnodes = np.where(((nodes == 0) | (nodes == p)).any(1))[0]
            L = np.array(N) * p
            lat = (cell[:, None, :] * p + nodes[self.bnodes][None]) % L
            key = (lat * np.cumprod(np.concatenate([[1], L[:-1]]))).sum(-1)
            uniq, inv = np.unique(key.reshape(-1), return_inverse=True)
            self.trace, self.T = inv.reshape(E, -1).astype(np.int64), len(uniq)
            self.orders, self.face_kind = np.full(E, p), None
            self.face_degree = np.zeros((E, 2 * d), dtype=np.int64)

    def handle(self, c):
        kw = dict(gamma=1.4, Pr=0.72, Re=_reynolds(c), Minf=0.2, alpha=ALPHA, precision=PREC[c["prec"]],
                  stab=1 if c["stab"] == "roe" else 0)
        if self.mixed:
            return iedg.MixedOrderMesh(self.X, self.trace, self.T, self.orders, self.face_degree,
                                       face_kind=self.face_kind, u_far=_far(c) if self.face_kind is not None else None,
                                       **kw)
        return iedg.Mesh(self.X, self.trace, self.T, int(c["p"]),
                         flags=iedg.FLAG_MASS_SCALING if c["scale"] else 0, **kw)


def _reynolds(c):
    return 1.0e3 if c["d"] == 2 or c["shape"] == "wall" else 2.5e5


def _far(c):
    return np.array([1.0, 0.5, 0.05] + [0.0] * (c["d"] - 2) + [1.0 / (1.4 * 0.4 * 0.04) + 0.5 * 0.2525])


# ---------------------------------------------------------------------------- states
def _field(c, seed, dev):
    """Conserved field of position [..., d]: 3D a Taylor-Green vortex with seeded phases;
    2D a free stream with seeded Fourier modes of 1 %."""
    g = torch.Generator().manual_seed(int(seed))
    d, p0 = c["d"], 1.0 / (1.4 * 0.04)
    ph = (2 * math.pi * torch.rand(3, generator=g, dtype=F64)).tolist()
    amp, phi = torch.rand(4, 9, generator=g, dtype=F64).to(dev) + 0.5, 6.28 * torch.rand(4, 9, generator=g, dtype=F64)
    phi, ks = phi.to(dev), torch.tensor([[a, b] for a in (1, 2, 3) for b in (1, 2, 3)], dtype=F64, device=dev)

    def f(x):
        if d == 3:
            X, Y, Z = (2 * math.pi * x[..., r] + ph[r] for r in range(3))
            v = [X.sin() * Y.cos() * Z.cos(), -X.cos() * Y.sin() * Z.cos(), 0 * X]
            pr = p0 + ((2 * X).cos() + (2 * Y).cos()) * ((2 * Z).cos() + 2.0) / 16.0
            rho = pr / p0
            return torch.stack([rho] + [rho * w for w in v] + [pr / 0.4 + 0.5 * rho * sum(w * w for w in v)], -1)
        arg = 2 * math.pi * x @ ks.T
        w = torch.stack([(amp[i] * (arg + phi[i]).sin()).mean(-1) for i in range(4)], -1)
        base = torch.tensor([1.0, 1.0, 0.0, p0 / 0.4 + 0.5], dtype=F64, device=dev)
        return base + 0.01 * w * torch.tensor([1.0, 1.0, 1.0, p0 / 0.4], dtype=F64, device=dev)
    return f


def _state(c, mesh, seed, dev):
    """u, q, uhat, u_ref, duhat; element arrays flat over all nodes, [nodes, m] and [nodes, m, d]."""
    f = _field(c, seed, dev)
    m = mesh.m
    gen = torch.Generator(device=dev).manual_seed(int(seed) + 1)

    def noise(*shape):
        return 2 * torch.rand(*shape, generator=gen, dtype=F64, device=dev) - 1

    X = np.concatenate(mesh.X) if mesh.mixed else mesh.X.reshape(-1, mesh.d)
    x = torch.as_tensor(X, device=dev)
    u = f(x)
    sigma = torch.ones(m, dtype=F64, device=dev)
    sigma[-1] = 1.0 / (1.4 * 0.4 * 0.04)
    h = 1e-5
    q = torch.stack([(f(x + h * e) - f(x - h * e)) / (2 * h)
                     for e in torch.eye(mesh.d, dtype=F64, device=dev)], -1).contiguous()
    u = u + 0.01 * sigma * noise(*u.shape)
    if mesh.mixed:
        # the field at one of the element slots that share the node, with noise of its own
        pos = np.zeros((mesh.T, mesh.d))
        for e in range(len(mesh.orders)):
            xi = _slot_points(mesh.d, int(mesh.orders[e]), mesh.face_degree[e])
            pos[mesh.trace[e]] = _tensor_basis(int(mesh.orders[e]), xi) @ mesh.X[e]
        uhat = f(torch.as_tensor(pos, device=dev))
        uhat = uhat + 0.01 * sigma * noise(*uhat.shape)
    else:
        E, Np = mesh.X.shape[:2]
        ub = u.reshape(E, Np, m)[:, torch.as_tensor(mesh.bnodes, device=dev)].reshape(-1, m).cpu().numpy()
        t = mesh.trace.reshape(-1)
        n = np.bincount(t, minlength=mesh.T)
        uhat = torch.as_tensor(np.stack([np.bincount(t, ub[:, i], mesh.T) / n for i in range(m)], -1), device=dev)
    u_ref = u + 0.01 * sigma * noise(*u.shape)
    duhat = 1e-3 * sigma * noise(mesh.T, m)
    return u, q, uhat.contiguous(), u_ref, duhat


def prepare(case, seed):
    mesh = _Mesh(case)
    h = mesh.handle(case)
    if case["precond"] == "bilu0":
        h.set_trace_precond(iedg.PREC_BILU0)
    u, q, uhat, u_ref, duhat = _state(case, mesh, seed, "cuda")
    s = {"case": case, "h": h, "u": u.reshape(h._ushape), "q": q.reshape(h._qshape), "uhat": uhat,
         "u_ref": u_ref.reshape(h._ushape), "duhat": duhat}
    if case["op"] == "trace":
        s["K"], s["R"] = h.assemble_condensed(s["u"], s["q"], uhat, u_ref=s["u_ref"])
    return s


def run(s):
    h, op = s["h"], s["case"]["op"]
    if op == "residual":
        return h.eval_residual(s["u"], s["uhat"], u_ref=s["u_ref"])
    if op == "trace":
        return {"dU": h.trace_solve(s["K"], s["R"], rtol=RTOL, max_iter=2000)[0]}
    out = h.eval_residual(s["u"], s["uhat"], q=s["q"], u_ref=s["u_ref"])
    out.pop("q")
    out["K"], out["R"] = h.assemble_condensed(s["u"], s["q"], s["uhat"], u_ref=s["u_ref"])
    dU = s["duhat"]
    if op == "iteration":
        dU = out["dU"] = h.trace_solve(out["K"], out["R"], rtol=RTOL, max_iter=2000)[0]
    out["du"], out["dq"] = h.back_substitute(dU)
    return out


def work(case):
    """Values in and out once; the partial LU of every element's bordered matrix and the
    sum-factorised assembly (the 1D contractions of its columns)."""
    mesh = _Mesh(case)
    d, m = mesh.d, mesh.m
    op = case["op"]
    byts = flops = pairs = 0.0
    for e, p in enumerate(mesh.orders.tolist()):
        Np, nq1 = (p + 1) ** d, p + 2
        Nb = len(mesh.trace[e])
        pairs += Nb * Nb
        byts += 8.0 * Np * (d + m * (2 + d)) + 8.0 * Np * m * (1 + 2 * d)        # X, u, u_ref, q; r_u, r_q, q out
        if op not in ("residual", "trace"):
            nu, n = m * Np, m * (Np + Nb)
            flops += sum(2.0 * (n - k - 1) * (n - k) for k in range(nu))
            col = sum((3 if r else 2) * (p + 1) ** (r + 1) * nq1 ** (d - r) for r in range(d)) / 2 + d * nq1 ** (d - 1)
            flops += 2.0 * m * m * (Np + Nb) * col
            byts += 8.0 * Np * m * (1 + d)                                        # du, dq
        else:
            flops += 2.0 * m * (1 + d) * 2 * (p + 1) * nq1 ** d * d
    byts += 8.0 * mesh.T * m * 3
    if op != "residual":
        # trace nodes shared by 2^k elements: distinct blocks, bounded below by the pairs' share
        nnzb = _nnzb(mesh) if mesh.T * 200 < 5e6 else 0.75 * pairs
        byts += 8.0 * nnzb * m * m
        flops += 2.0 * nnzb * m * m if op in ("trace", "iteration") else 0.0
    return {"bytes": byts, "flops": flops}


def _nnzb(mesh):
    return len(np.unique(np.concatenate([(t[:, None] * mesh.T + t[None, :]).reshape(-1) for t in mesh.trace])))


# ------------------------------------------------------------------ exact: 1D and tensor tables
def _lagrange(p, x):
    """[len(x), p+1] values and derivatives of the degree-p Gauss-Lobatto basis."""
    nodes = workloads.gll_positions(p)
    x = np.asarray(x, dtype=np.float64)
    c = np.array([[np.prod([x[g] - nodes[k] for k in range(p + 1) if k != j]) for j in range(p + 1)]
                  for g in range(len(x))])
    w = np.array([np.prod([nodes[j] - nodes[k] for k in range(p + 1) if k != j]) for j in range(p + 1)])
    dv = np.array([[sum(np.prod([x[g] - nodes[k] for k in range(p + 1) if k not in (j, s)])
                        for s in range(p + 1) if s != j) for j in range(p + 1)] for g in range(len(x))])
    return c / w, dv / w


def _tensor_basis(p, pts, der=None):
    """[len(pts), (p+1)^d] basis at reference points, or its derivative in direction `der`."""
    d = pts.shape[1]
    idx, out = _multi(p + 1, d), np.ones((len(pts), (p + 1) ** d))
    for r in range(d):
        V, D = _lagrange(p, pts[:, r])
        out *= (D if r == der else V)[:, idx[:, r]]
    return out


def _face_points(d, f, t):
    """Face points from tangential coordinates t [n, d-1] (first tangential direction first)."""
    return np.insert(t, f // 2, 1.0 if f % 2 else -1.0, axis=1)


def _slot_points(d, p, deg):
    """Reference positions of an element's trace slots."""
    nodes = _multi(p + 1, d)
    on = np.zeros(len(nodes), dtype=bool)
    for f in range(2 * d):
        if deg[f] == 0:
            on |= nodes[:, f // 2] == (p if f % 2 else 0)
    out = [workloads.gll_positions(p)[nodes[on]]]
    for f in range(2 * d):
        if deg[f]:
            out.append(_face_points(d, f, workloads.gll_positions(int(deg[f]))[_multi(int(deg[f]) + 1, d - 1)]))
    return np.concatenate(out)


def _slot_basis(d, p, deg, fpts, fphi, t1):
    """[Nfp, Nb_e] trace basis at the face points: on a continuous face the element basis
    of its nodes, on a face of degree q the degree-q basis of its private nodes."""
    nodes, nf, Nfq = _multi(p + 1, d), 2 * d, len(t1)
    face = np.repeat(np.arange(nf), Nfq)
    on = np.stack([nodes[:, f // 2] == (p if f % 2 else 0) for f in range(nf)])
    edg = [f for f in range(nf) if deg[f] == 0]
    keep = on[edg].any(0) if edg else np.zeros(len(nodes), dtype=bool)
    mu = [fphi[:, keep] * np.isin(face, edg)[:, None]]
    for f in range(nf):
        if deg[f]:
            blk = np.zeros((nf * Nfq, (int(deg[f]) + 1) ** (d - 1)))
            blk[face == f] = _tensor_basis(int(deg[f]), t1)
            mu.append(blk)
    return np.concatenate(mu, 1)


# ------------------------------------------------------------------ exact: pointwise physics
def _physics(c):
    g, Pr, Re, d = 1.4, 0.72, _reynolds(c), c["d"]

    def parts(u):
        v = u[1:d + 1] / u[0]
        return v, (g - 1) * (u[-1] - 0.5 * u[0] * (v @ v))

    def flux(u, q):
        v, p = parts(u)
        E = u[-1] / u[0]
        dv = (q[1:d + 1] - v[:, None] * q[0]) / u[0]
        de = (q[-1] - E * q[0]) / u[0] - v @ dv
        eye = torch.eye(d, dtype=u.dtype, device=u.device)
        tau = (dv + dv.T - (2.0 / 3.0) * torch.trace(dv) * eye) / Re
        mom = torch.outer(u[1:d + 1], v) + p * eye - tau
        return torch.cat([u[1:d + 1][None], mom, (v * (u[-1] + p) - g / (Re * Pr) * de - v @ tau)[None]])

    def lam(u, n):
        v, p = parts(u)
        return torch.abs(v @ n) + torch.sqrt(g * p / u[0])

    def waves(uh, x, n):
        """A_n x and |A_n| x of the Euler flux at uh."""
        v, p = parts(uh)
        c2, vn, H = g * p / uh[0], v @ n, (uh[-1] + p) / uh[0]
        cs = torch.sqrt(c2)
        dp = (g - 1) * (x[-1] - v @ x[1:d + 1] + 0.5 * (v @ v) * x[0])
        rdv = n @ x[1:d + 1] - vn * x[0]
        one = torch.ones_like(vn)[None]
        rm = torch.cat([one, v - cs * n, (H - cs * vn)[None]])
        rp = torch.cat([one, v + cs * n, (H + cs * vn)[None]])
        am, ap = (dp - cs * rdv) / (2 * c2), (dp + cs * rdv) / (2 * c2)
        rest = x - am * rm - ap * rp
        A = vn * rest + (vn - cs) * am * rm + (vn + cs) * ap * rp
        S = torch.abs(vn) * rest + torch.abs(vn - cs) * am * rm + torch.abs(vn + cs) * ap * rp
        return A, S

    def fhat(uh, u, q, n):
        s = waves(uh, u - uh, n)[1] if c["stab"] == "roe" else lam(uh, n) * (u - uh)
        return flux(uh, q) @ n + s

    far = torch.as_tensor(_far(c))

    def bhat(uh, u, q, n, kind):
        a, s = waves(uh, uh - u, n)
        a2, s2 = waves(uh, uh - far.to(uh.device), n)
        fh = fhat(uh, u, q, n)
        wall = torch.cat([(uh[0] - u[0])[None], uh[1:d + 1], fh[-1][None]])
        return torch.where(kind == 1, 0.5 * (a + s) + 0.5 * (a2 - s2), torch.where(kind == 2, wall, fh))

    return flux, fhat, bhat


def _values_and_jacobians(fun, args, n_diff):
    """fun over points (vmap) and its Jacobians in the first n_diff arguments."""
    vals = torch.func.vmap(fun)(*args)
    jac = torch.func.vmap(torch.func.jacfwd(fun, argnums=tuple(range(n_diff))))(*args)
    return vals, jac


# ------------------------------------------------------------------ exact: elements
def _elements(c, mesh, els, st, dev, want):
    """Residuals, condensed blocks and updates of the elements `els` (equal order)."""
    d, m, p = mesh.d, mesh.m, int(mesh.orders[els[0]])
    u, q, uh, ur, dU = st                                  # [n, Np, ..], trace values [n, Nb, m]
    n, Np, nf = len(els), (p + 1) ** d, 2 * d
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=dev)  # noqa: E731
    x1, w1 = np.polynomial.legendre.leggauss(p + 2)
    gi, ti = _multi(p + 2, d), _multi(p + 2, d - 1)
    fp = np.concatenate([_face_points(d, f, x1[ti]) for f in range(nf)])
    phi, fphi = T(_tensor_basis(p, x1[gi])), T(_tensor_basis(p, fp))
    dphi = T(np.stack([_tensor_basis(p, x1[gi], r) for r in range(d)]))
    dfphi = T(np.stack([_tensor_basis(p, fp, r) for r in range(d)]))
    if mesh.mixed:
        mus = [_slot_basis(d, p, mesh.face_degree[e], fp, fphi.cpu().numpy(), x1[ti]) for e in els]
        Nb = max(x.shape[1] for x in mus)
        mu = T(np.stack([np.pad(x, ((0, 0), (0, Nb - x.shape[1]))) for x in mus]))
    else:
        mu = fphi[:, T(mesh.bnodes)][None].expand(n, -1, -1)
        Nb = mu.shape[2]
    X = T(np.stack([mesh.X[e] for e in els]))
    J = torch.einsum("rga,eai->egir", dphi, X)
    w = torch.linalg.det(J) * T(w1[gi].prod(1))
    gphi = torch.einsum("rga,egrj->ejga", dphi, torch.linalg.inv(J))
    Jf = torch.einsum("rga,eai->egir", dfphi, X)
    nref = np.zeros((nf, d))
    for f in range(nf):
        nref[f, f // 2] = 1.0 if f % 2 else -1.0
    nds = torch.einsum("egri,gr->egi", torch.linalg.inv(Jf) * torch.linalg.det(Jf)[..., None, None],
                       T(np.repeat(nref, len(ti), 0)))
    area = torch.linalg.norm(nds, dim=-1)
    wf, nrm = area * T(np.tile(w1[ti].prod(1), nf)), nds / area[..., None]
    M = torch.einsum("eg,ga,gb->eab", w, phi, phi)
    B = torch.einsum("eg,ejga,gb->ejab", w, gphi, phi)
    En = torch.einsum("eg,egj,ga,egt->ejat", wf, nrm, fphi, mu)
    G, H = torch.linalg.solve(M[:, None], B), torch.linalg.solve(M[:, None], En)
    qs = torch.einsum("ejat,eti->eaij", H, uh) - torch.einsum("ejab,ebi->eaij", G, u)
    out = {}
    if q is None:
        q = out["q"] = qs
        out["r_q"] = torch.zeros_like(qs)
    else:
        out["r_q"] = torch.einsum("eab,ebij->eaij", M, q - qs)
    flux, fhat, bhat = _physics(c)
    at = lambda tab, v: torch.einsum("ga,ea...->eg...", tab, v)  # noqa: E731
    flat = lambda v: v.reshape(-1, *v.shape[2:])  # noqa: E731
    un = lambda v: v.reshape(n, -1, *v.shape[1:])  # noqa: E731
    uf, uhf = at(fphi, u), torch.einsum("egt,eti->egi", mu, uh)
    kind = None
    if mesh.face_kind is not None:
        kind = T(np.repeat(np.stack([mesh.face_kind[e] for e in els]), len(ti), 1))

    def residual(qq):
        F = un(torch.func.vmap(flux)(flat(at(phi, u)), flat(at(phi, qq))))
        args = [flat(uhf), flat(uf), flat(at(fphi, qq)), flat(nrm)]
        fh = un(torch.func.vmap(fhat)(*args))
        ft = fh if kind is None else un(torch.func.vmap(bhat)(*args, kind.reshape(-1)))
        ru = (ALPHA * torch.einsum("eab,ebi->eai", M, u - ur) - torch.einsum("eg,egij,ejga->eai", w, F, gphi)
              + torch.einsum("eg,egi,ga->eai", wf, fh, fphi))
        return ru, torch.einsum("eg,egi,egt->eti", wf, ft, mu)

    out["r_u"], out["rhat"] = residual(q)
    if not want:
        return out
    # Newton blocks with the gradient eliminated (fluxes are affine in q)
    Fs, Gs = residual(qs)
    _, (Fu, Fq) = _values_and_jacobians(flux, (flat(at(phi, u)), flat(at(phi, q))), 2)
    args = (flat(uhf), flat(uf), flat(at(fphi, q)), flat(nrm))
    _, (fuh, fu, fq) = _values_and_jacobians(fhat, args, 3)
    wJ = w[:, None, :, None] * gphi
    Fu, Fq, fuh, fu, fq = (un(v) for v in (Fu, Fq, fuh, fu, fq))
    tf = (fuh, fu, fq)
    if kind is not None:
        tf = tuple(un(v) for v in _values_and_jacobians(bhat, args + (kind.reshape(-1),), 3)[1])

    def rows(test_f, fuh, fu, fq, volume):
        """Rows of the element system for face tests `test_f` [n, Nfp, rows] (and the volume)."""
        R = test_f.shape[2]
        wt = wf[..., None] * test_f                                          # [n, Nfp, rows]
        uq = torch.einsum("egr,egikl->eiklrg", wt, fq) @ fphi                # [n, i, k, l, rows, Np]
        uu = torch.einsum("egr,egik->eikrg", wt, fu) @ fphi
        if volume:
            uq = uq - torch.einsum("ejga,egijkl->eiklag", wJ, Fq) @ phi
            uu = uu - torch.einsum("ejga,egijk->eikag", wJ, Fu) @ phi
        uh_ = torch.einsum("egr,egik->eikrg", wt, fuh) @ mu[:, None, None]
        uu = uu - sum(uq[:, :, :, j] @ G[:, j][:, None, None] for j in range(d))
        uh_ = uh_ + sum(uq[:, :, :, j] @ H[:, j][:, None, None] for j in range(d))
        return (uu.permute(0, 1, 3, 2, 4).reshape(n, m * R, m * Np),
                uh_.permute(0, 1, 3, 2, 4).reshape(n, m * R, m * Nb))

    At, Bt = rows(fphi[None].expand(n, -1, -1), fuh, fu, fq, True)
    At = At + ALPHA * torch.block_diag(*[torch.ones(1, 1, dtype=F64, device=dev)] * m)[None, :, None, :, None].mul(
        M[:, None, :, None, :]).reshape(n, m * Np, m * Np)
    Ct, Dt = rows(mu, *tf, False)
    Ft, Gt = (-v.transpose(1, 2).reshape(n, -1) for v in (Fs, Gs))
    sol = torch.linalg.solve(At, torch.cat([Bt, Ft[..., None]], 2))
    S = torch.cat([Dt, Gt[..., None]], 2) - Ct @ sol
    out["K"] = S[..., :-1].reshape(n, m, Nb, m, Nb).permute(0, 2, 4, 1, 3)   # [n, s, t, i, k]
    out["R"] = S[..., -1].reshape(n, m, Nb).transpose(1, 2)

    def update(dU):
        du = sol[..., -1] - torch.einsum("eab,eb->ea", sol[..., :-1], dU.transpose(1, 2).reshape(n, -1))
        du = du.reshape(n, m, Np).transpose(1, 2)
        return du, (qs - q - torch.einsum("ejab,ebi->eaij", G, du) + torch.einsum("ejat,eti->eaij", H, dU))

    if dU is None:
        out["update"] = update
    else:
        out["du"], out["dq"] = update(dU)
    return out


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    mesh, op = _Mesh(case), case["op"]
    E, d, m = len(mesh.orders), mesh.d, mesh.m
    if op in ("trace", "iteration") and mesh.T * m > 22000:
        return None                # the dense solve of the trace system would take too long
    u, q, uhat, u_ref, duhat = _state(case, mesh, seed, dev)
    npe = (mesh.orders + 1) ** d
    off = np.concatenate([[0], np.cumsum(npe)])
    want, solve = op != "residual", op in ("trace", "iteration")
    rows = torch.as_tensor(np.concatenate([np.repeat(t, len(t)) for t in mesh.trace]), device=dev)
    if want:
        cols = torch.as_tensor(np.concatenate([np.tile(t, len(t)) for t in mesh.trace]), device=dev)
        uniq, inv = torch.unique(rows * mesh.T + cols, return_inverse=True)
        poff = np.concatenate([[0], np.cumsum([len(t) ** 2 for t in mesh.trace])])
        K = torch.zeros(len(uniq), m, m, dtype=F64, device=dev)
    R, rfl = (torch.zeros(mesh.T, m, dtype=F64, device=dev) for _ in range(2))
    res = {"r_q": torch.empty_like(q), "r_u": torch.empty_like(u)}
    if op == "residual":
        res["q"] = torch.empty_like(q)
    elif op != "trace":
        res["du"], res["dq"] = torch.empty_like(u), torch.empty_like(q)
    later = []
    for p in sorted(set(mesh.orders.tolist())):
        group = np.where(mesh.orders == p)[0]
        per = max(1, int(3e9 / (8.0 * (p + 1) ** d * (p + 2) ** d * m * m * d * 3)))
        for els in np.array_split(group, -(-len(group) // per)):
            nodes = torch.as_tensor((off[els][:, None] + np.arange((p + 1) ** d)).reshape(-1), device=dev)
            Nb = max(len(mesh.trace[e]) for e in els)
            tr = np.zeros((len(els), Nb), dtype=np.int64)
            ok = np.zeros((len(els), Nb), dtype=bool)
            for k, e in enumerate(els):
                tr[k, :len(mesh.trace[e])], ok[k, :len(mesh.trace[e])] = mesh.trace[e], True
            tr, okt = torch.as_tensor(tr, device=dev), torch.as_tensor(ok, device=dev)
            el = lambda v: v[nodes].reshape(len(els), -1, *v.shape[1:])  # noqa: E731
            tv = lambda v: v[tr] * okt[..., None]  # noqa: E731
            o = _elements(case, mesh, els, (el(u), None if op == "residual" else el(q), tv(uhat), el(u_ref),
                                            None if solve else tv(duhat)), dev, want)
            for k in ("r_q", "r_u", "q", "du", "dq"):
                if k in o and k in res:
                    res[k][nodes] = o[k].reshape(-1, *o[k].shape[2:])
            rfl.index_add_(0, tr[okt], o["rhat"][okt])
            if want:
                R.index_add_(0, tr[okt], o["R"][okt])
                at = torch.as_tensor(np.concatenate([np.arange(poff[e], poff[e + 1]) for e in els]), device=dev)
                both = okt[:, :, None] & okt[:, None, :]
                K.index_add_(0, inv[at], o["K"][both])
            if solve:
                later.append((nodes, tr, okt, o["update"]))
    if op == "residual":
        return {"q": res["q"], "r_q": res["r_q"], "r_u": res["r_u"], "r_fl": rfl}
    dU = duhat
    if solve:
        r, t = uniq // mesh.T, uniq % mesh.T
        D = torch.zeros(mesh.T, m, mesh.T, m, dtype=F64, device=dev)
        D[r, :, t] = K
        dU = torch.linalg.solve(D.reshape(mesh.T * m, -1), R.reshape(-1)).reshape(mesh.T, m)
        if op == "trace":
            return {"dU": dU}
        for nodes, tr, okt, update in later:
            du, dq = update(dU[tr] * okt[..., None])
            res["du"][nodes], res["dq"][nodes] = du.reshape(-1, m), dq.reshape(-1, m, d)
    out = {"r_q": res["r_q"], "r_u": res["r_u"], "r_fl": rfl, "K": K, "R": R, "du": res["du"], "dq": res["dq"]}
    if op == "iteration":
        out["dU"] = dU
    return out
