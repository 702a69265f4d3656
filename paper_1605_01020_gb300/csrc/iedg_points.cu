// Quadrature-point physics and residual of the IEDG weak form.
//
//  * Navier-Stokes flux F(u, q) (Sec. 2.1): inviscid part rho v_j, rho v_i v_j +
//    delta_ij p, v_j (rho E + p); viscous part tau_ij = (1/Re)(d_j v_i + d_i v_j -
//    2/3 delta_ij d_k v_k); heat term (gamma / (Re Pr)) d_j e with e = E - |v|^2/2,
//    taken with the dissipative sign (the energy flux loses v_i tau_ij + it).
//  * Lax-Friedrichs numerical flux (Eq. IEDG d): fhat = F(uhat, q) n + lambda (u -
//    uhat), lambda = |vhat . n| + chat evaluated at uhat.
//  * Pointwise Jacobians by forward-mode dual numbers, m directions per pass:
//    one pass over u (or uhat), one pass per gradient direction l over q_{., l}.
//  * Residual projections (Eq. IEDG b, c), in 3D as sums over one direction at a time:
//      R_u[a][i]  = sum_{g,r} Dxi_r[g][a] fvol[i][r][g] + sum_g Phi[g][a] mvol[i][g]
//                 + sum_fp PhiF[fp][a] fsur[i][fp]
//      Rhat[s][i] = sum_fp PhiF[fp][bnode[s]] fsur[i][fp]
//    with fvol = -w Jinv[r][j] F_ij, mvol = alpha w (u - u_ref)_i, fsur = wf fhat_i.
//  * R_q = M (q - q*) where q* = H_l uhat - G_l u is the lifted gradient that makes
//    R_q vanish (Eq. IEDG a is linear: R_q = M q + B_l u - E_l uhat).
#include <type_traits>

#include "iedg_internal.cuh"

namespace iedg {
namespace {

// ------------------------------------------------------------------ dual numbers
template <int N>
struct Dual {
  double v;
  double t[N];
};

template <int N>
__device__ inline Dual<N> mkconst(double v) {
  Dual<N> r;
  r.v = v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.t[k] = 0.0;
  return r;
}
template <int N>
__device__ inline Dual<N> operator+(const Dual<N>& a, const Dual<N>& b) {
  Dual<N> r; r.v = a.v + b.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.t[k] = a.t[k] + b.t[k];
  return r;
}
template <int N>
__device__ inline Dual<N> operator-(const Dual<N>& a, const Dual<N>& b) {
  Dual<N> r; r.v = a.v - b.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.t[k] = a.t[k] - b.t[k];
  return r;
}
template <int N>
__device__ inline Dual<N> operator*(const Dual<N>& a, const Dual<N>& b) {
  Dual<N> r; r.v = a.v * b.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.t[k] = a.t[k] * b.v + a.v * b.t[k];
  return r;
}
template <int N>
__device__ inline Dual<N> operator*(double a, const Dual<N>& b) {
  Dual<N> r; r.v = a * b.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.t[k] = a * b.t[k];
  return r;
}
template <int N>
__device__ inline Dual<N> operator+(const Dual<N>& a, double b) {
  Dual<N> r = a; r.v += b; return r;
}
template <int N>
__device__ inline Dual<N> recip(const Dual<N>& a) {
  Dual<N> r; r.v = 1.0 / a.v;
  double s = -r.v * r.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.t[k] = s * a.t[k];
  return r;
}
template <int N>
__device__ inline Dual<N> dsqrt(const Dual<N>& a) {
  Dual<N> r; r.v = sqrt(a.v);
  double s = 0.5 / r.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.t[k] = s * a.t[k];
  return r;
}
template <int N>
__device__ inline Dual<N> dabs(const Dual<N>& a) {
  double s = a.v > 0 ? 1.0 : (a.v < 0 ? -1.0 : 0.0);   // sign(0) := 0
  Dual<N> r; r.v = fabs(a.v);
#pragma unroll
  for (int k = 0; k < N; ++k) r.t[k] = s * a.t[k];
  return r;
}
// double with dual: as a dual of zero tangent would give, its products rounded before a sum
template <int N>
__device__ inline Dual<N> operator*(const Dual<N>& a, double b) {
  Dual<N> r; r.v = a.v * b;
#pragma unroll
  for (int k = 0; k < N; ++k) r.t[k] = __dmul_rn(a.t[k], b);
  return r;
}
template <int N>
__device__ inline Dual<N> times(double a, const Dual<N>& b) {
  Dual<N> r; r.v = a * b.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.t[k] = __dmul_rn(a, b.t[k]);
  return r;
}
__device__ inline double times(double a, double b) { return a * b; }
template <int N>
__device__ inline Dual<N> times(const Dual<N>& a, const Dual<N>& b) { return a * b; }
template <int N>
__device__ inline Dual<N> operator-(double a, const Dual<N>& b) {
  Dual<N> r; r.v = a - b.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.t[k] = 0.0 - b.t[k];
  return r;
}
template <int N>
__device__ inline Dual<N> operator+(double a, const Dual<N>& b) {
  Dual<N> r = b; r.v = a + b.v; return r;
}
__device__ inline double recip(double a) { return 1.0 / a; }
__device__ inline double dsqrt(double a) { return sqrt(a); }
__device__ inline double dabs(double a) { return fabs(a); }
template <class T> __device__ inline T mk(double v);
template <> __device__ inline double mk<double>(double v) { return v; }
template <> __device__ inline Dual<4> mk<Dual<4>>(double v) { return mkconst<4>(v); }
template <> __device__ inline Dual<5> mk<Dual<5>>(double v) { return mkconst<5>(v); }

// Navier-Stokes flux F[i][j], i < M = D + 2, j < D.  u and q may be of different types: with
// u = double and q = Dual the inviscid part and everything else that depends on u alone is
// evaluated once without tangents (the result has the bits of the all-dual evaluation).
template <int D, class TU, class T>
__device__ void ns_flux(const TU* u, const T (*q)[D], const Phys& ph, T (*F)[D]) {
  constexpr int M = D + 2;
  const TU rinv = recip(u[0]);
  TU v[D];
#pragma unroll
  for (int i = 0; i < D; ++i) v[i] = u[1 + i] * rinv;
  const TU E = u[M - 1] * rinv;
  TU vv = v[0] * v[0];
#pragma unroll
  for (int i = 1; i < D; ++i) vv = vv + v[i] * v[i];
  const TU p = (ph.gamma - 1.0) * (u[M - 1] - 0.5 * (u[0] * vv));
  T dv[D][D];
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int j = 0; j < D; ++j) dv[i][j] = (q[1 + i][j] - times(v[i], q[0][j])) * rinv;
  T div = dv[0][0];
#pragma unroll
  for (int k = 1; k < D; ++k) div = div + dv[k][k];
  const double ire = 1.0 / ph.Re, kap = ph.gamma / (ph.Re * ph.Pr);
#pragma unroll
  for (int j = 0; j < D; ++j) {
    T de = (q[M - 1][j] - times(E, q[0][j])) * rinv;
#pragma unroll
    for (int k = 0; k < D; ++k) de = de - times(v[k], dv[k][j]);
    if constexpr (std::is_same<TU, T>::value) F[0][j] = u[1 + j];
    else F[0][j] = mk<T>(u[1 + j]);
    T fe = v[j] * (u[M - 1] + p) - kap * de;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      T tau = dv[i][j] + dv[j][i];
      if (i == j) tau = tau - (2.0 / 3.0) * div;
      tau = ire * tau;
      T fm = u[1 + i] * v[j] - tau;
      if (i == j) fm = fm + p;
      F[1 + i][j] = fm;
      fe = fe - times(v[i], tau);
    }
    F[M - 1][j] = fe;
  }
}

template <int D, class T>
__device__ T lf_lambda(const T* u, const double* n, const Phys& ph) {
  constexpr int M = D + 2;
  const T rinv = recip(u[0]);
  T vn = mk<T>(0.0), vv = mk<T>(0.0);
#pragma unroll
  for (int j = 0; j < D; ++j) {
    T vj = u[1 + j] * rinv;
    vn = vn + n[j] * vj;
    vv = vv + vj * vj;
  }
  T p = (ph.gamma - 1.0) * (u[M - 1] - 0.5 * (u[0] * vv));
  return dabs(vn) + dsqrt((ph.gamma * p) * rinv);
}

// Roe-type stabilisation out = |A_n(uh)| du, A_n the normal Jacobian of the Euler flux
// at uh (Sec. 2.1).  Eigenvalues v_n - c, v_n (d-fold), v_n + c; the acoustic waves of
// du have strengths a_-+ = (dp -+ c rho dv_n) / (2 c^2), with the linearised jumps
// dp = (gamma-1)(d(rhoE) - v.d(rho v) + |v|^2/2 drho), rho dv_n = n.d(rho v) - v_n drho,
// and eigenvectors (1, v -+ c n, H -+ c v_n); all other waves move at v_n:
//   |A_n| du = |v_n| du + (|v_n - c| - |v_n|) a_- r_- + (|v_n + c| - |v_n|) a_+ r_+ .
// T = double, or Dual<M> to differentiate with respect to uh (du may depend on it).
template <int D, class T>
__device__ void roe_apply(const T* uh, const T* du, const double* n, const Phys& ph, T* out) {
  constexpr int M = D + 2;
  const T rinv = recip(uh[0]);
  T v[D];
#pragma unroll
  for (int j = 0; j < D; ++j) v[j] = uh[1 + j] * rinv;
  T vn = mk<T>(0.0), q2 = mk<T>(0.0), vdm = mk<T>(0.0), ndm = mk<T>(0.0);
#pragma unroll
  for (int j = 0; j < D; ++j) {
    vn = vn + n[j] * v[j];
    q2 = q2 + v[j] * v[j];
    vdm = vdm + v[j] * du[1 + j];
    ndm = ndm + n[j] * du[1 + j];
  }
  const T p = (ph.gamma - 1.0) * (uh[M - 1] + (-0.5) * (uh[0] * q2));
  const T c2 = ph.gamma * (p * rinv);
  const T c = dsqrt(c2);
  const T H = (uh[M - 1] + p) * rinv;
  const T dp = (ph.gamma - 1.0) * (du[M - 1] + (-1.0) * vdm + 0.5 * (q2 * du[0]));
  const T rdvn = ndm + (-1.0) * (vn * du[0]);
  const T ic2 = 0.5 * recip(c2);
  const T am = (dp + (-1.0) * (c * rdvn)) * ic2;
  const T ap = (dp + c * rdvn) * ic2;
  const T l0 = dabs(vn);
  const T wm = (dabs(vn + (-1.0) * c) + (-1.0) * l0) * am;
  const T wp = (dabs(vn + c) + (-1.0) * l0) * ap;
  out[0] = l0 * du[0] + wm + wp;
#pragma unroll
  for (int j = 0; j < D; ++j) out[1 + j] = l0 * du[1 + j] + wm * (v[j] + (-n[j]) * c) + wp * (v[j] + n[j] * c);
  out[M - 1] = l0 * du[M - 1] + wm * (H + (-1.0) * (c * vn)) + wp * (H + c * vn);
}

// out = A_n(uh) x, A_n = d(F_inv . n)/du the normal Jacobian of the Euler flux at uh,
// from the differentials of rho v_n, rho v v_n + p n, (rho E + p) v_n with
// dp = (gamma-1)(x_E - v.x_m + |v|^2/2 x_rho) and H = (rho E + p)/rho.
template <int D, class T>
__device__ void normal_jac_apply(const T* uh, const T* x, const double* n, const Phys& ph, T* out) {
  constexpr int M = D + 2;
  const T rinv = recip(uh[0]);
  T v[D];
#pragma unroll
  for (int j = 0; j < D; ++j) v[j] = uh[1 + j] * rinv;
  T vn = mk<T>(0.0), q2 = mk<T>(0.0), vdm = mk<T>(0.0), ndm = mk<T>(0.0);
#pragma unroll
  for (int j = 0; j < D; ++j) {
    vn = vn + n[j] * v[j];
    q2 = q2 + v[j] * v[j];
    vdm = vdm + v[j] * x[1 + j];
    ndm = ndm + n[j] * x[1 + j];
  }
  const T p = (ph.gamma - 1.0) * (uh[M - 1] + (-0.5) * (uh[0] * q2));
  const T H = (uh[M - 1] + p) * rinv;
  const T dp = (ph.gamma - 1.0) * (x[M - 1] + (-1.0) * vdm + 0.5 * (q2 * x[0]));
  out[0] = ndm;
#pragma unroll
  for (int j = 0; j < D; ++j) out[1 + j] = x[1 + j] * vn + v[j] * ndm + (-1.0) * (v[j] * (vn * x[0])) + n[j] * dp;
  out[M - 1] = (x[M - 1] + dp) * vn + H * (ndm + (-1.0) * (vn * x[0]));
}

// Far-field boundary flux (Sec. 2.1): bhat = (A_n + |A_n|)/2 (uh - u) + (A_n - |A_n|)/2
// (uh - u_b), A_n and |A_n| at uh.  T = double or Dual<M> (uh seeded; u, u_b constant).
template <int D, class T>
__device__ void farfield_flux(const T* uh, const double* u, const double* ub, const double* n, const Phys& ph,
                              T* b) {
  constexpr int M = D + 2;
  T a[M], c[M], Aa[M], Sa[M], Ac[M], Sc[M];
#pragma unroll
  for (int i = 0; i < M; ++i) {
    a[i] = uh[i] + mk<T>(-u[i]);
    c[i] = uh[i] + mk<T>(-ub[i]);
  }
  normal_jac_apply<D, T>(uh, a, n, ph, Aa);
  roe_apply<D, T>(uh, a, n, ph, Sa);
  normal_jac_apply<D, T>(uh, c, n, ph, Ac);
  roe_apply<D, T>(uh, c, n, ph, Sc);
#pragma unroll
  for (int i = 0; i < M; ++i) b[i] = 0.5 * (Aa[i] + Sa[i]) + 0.5 * (Ac[i] + (-1.0) * Sc[i]);
}

// Boundary flux of the trace equation at one face point of kind fk (far field or
// no-slip adiabatic wall): wf bhat into bval[M] and, with jac, the point's entries of
// Jb.  A wall's energy row is the energy row of fhat, whose derivatives the calling
// thread wrote to Jf, Su / lamw just before; they are read back here.
template <int D, int STAB>
__device__ __noinline__ void boundary_point(int fk, const double* uh, const double* u, const double* n, double wf,
                                            const Phys& ph, double fhatE, bool jac, const PointJac& PJ, int64_t e,
                                            int fp, int Nfp, double* bval) {
  constexpr int M = D + 2, NC = 2 + D;
  const size_t jfs = (size_t)(1 + D) * Nfp;
  auto jb = [&](int i, int k, int c) -> size_t { return (((size_t)(e * M + i) * M + k) * NC + c) * Nfp + fp; };
  auto put = [&](int i, int k, int c, double v) {
    PJ.Jb[jb(i, k, c)] = v;
    if (PJ.Jb32) PJ.Jb32[jb(i, k, c)] = (float)v;
  };
  if (fk == kFaceFarField) {
    double b[M];
    farfield_flux<D, double>(uh, u, ph.ub, n, ph, b);
#pragma unroll
    for (int i = 0; i < M; ++i) bval[i] = wf * b[i];
    if (!jac) return;
    Dual<M> ud[M], bd[M];
#pragma unroll
    for (int k = 0; k < M; ++k) { ud[k] = mkconst<M>(uh[k]); ud[k].t[k] = 1.0; }
    farfield_flux<D, Dual<M>>(ud, u, ph.ub, n, ph, bd);
#pragma unroll 1
    for (int k = 0; k < M; ++k) {
      double ek[M], Ak[M], Sk[M];
#pragma unroll
      for (int i = 0; i < M; ++i) ek[i] = (i == k) ? 1.0 : 0.0;
      normal_jac_apply<D, double>(uh, ek, n, ph, Ak);
      roe_apply<D, double>(uh, ek, n, ph, Sk);
#pragma unroll
      for (int i = 0; i < M; ++i) {
        put(i, k, 0, wf * bd[i].t[k]);
        put(i, k, 1, -0.5 * wf * (Ak[i] + Sk[i]));
#pragma unroll
        for (int l = 0; l < D; ++l) put(i, k, 2 + l, 0.0);
      }
    }
    return;
  }
  // wall: (rhohat - rho, rho vhat, fhat_E)
  bval[0] = wf * (uh[0] - u[0]);
#pragma unroll
  for (int j = 0; j < D; ++j) bval[1 + j] = wf * uh[1 + j];
  bval[M - 1] = wf * fhatE;
  if (!jac) return;
  const double* jfE = PJ.Jf + ((size_t)e * M * M + (size_t)(M - 1) * M) * jfs;   // row E of this element
#pragma unroll 1
  for (int k = 0; k < M; ++k) {
    for (int i = 0; i < M - 1; ++i) {
      put(i, k, 0, (i == k) ? wf : 0.0);
      put(i, k, 1, (i == 0 && k == 0) ? -wf : 0.0);
      for (int l = 0; l < D; ++l) put(i, k, 2 + l, 0.0);
    }
    const double* o = jfE + (size_t)k * jfs;
    put(M - 1, k, 0, o[fp]);
    double su;
    if constexpr (STAB == 1) su = PJ.Su[((size_t)(e * M + (M - 1)) * M + k) * Nfp + fp];
    else su = (k == M - 1) ? PJ.lamw[e * Nfp + fp] : 0.0;
    put(M - 1, k, 1, su);
    for (int l = 0; l < D; ++l) put(M - 1, k, 2 + l, o[(size_t)(1 + l) * Nfp + fp]);
  }
}

// The flux Jacobians at (u, q) by forward-mode duals, handed to the caller pass by pass
// so that no full dF / dQ array is held: on_u(Fd) after the pass over u, with
// Fd[i][j].t[k] = dF_ij/du_k, then on_q(l, Fd) after the pass over q_{., l}, with
// Fd[i][j].t[k] = dF_ij/dq_kl.
template <int D, class OnU, class OnQ>
__device__ __forceinline__ void flux_jacobians(const double* u, const double (*q)[D], const Phys& ph, OnU on_u,
                                               OnQ on_q) {
  constexpr int M = D + 2;
  using TD = Dual<M>;
  TD ud[M], qd[M][D], Fd[M][D];
  // pass over u
#pragma unroll
  for (int k = 0; k < M; ++k) { ud[k] = mkconst<M>(u[k]); ud[k].t[k] = 1.0; }
#pragma unroll
  for (int k = 0; k < M; ++k)
#pragma unroll
    for (int l = 0; l < D; ++l) qd[k][l] = mkconst<M>(q[k][l]);
  ns_flux<D, TD, TD>(ud, qd, ph, Fd);
  on_u(Fd);
  // passes over q_{., l}
#pragma unroll 1
  for (int l = 0; l < D; ++l) {
#pragma unroll
    for (int k = 0; k < M; ++k)
#pragma unroll
      for (int ll = 0; ll < D; ++ll) {
        qd[k][ll] = mkconst<M>(q[k][ll]);
        if (ll == l) qd[k][ll].t[k] = 1.0;
      }
    ns_flux<D, double, TD>(u, qd, ph, Fd);
    on_q(l, Fd);
  }
}

// ------------------------------------------------------------------ point kernels
// One CTA per element each.  k_point_res: the residual at (u, q), or at (u, q*) with the
// opposite sign into the right-hand sides of the bordered element matrices.  k_point_jac:
// the Jacobians at (u, q) into PointJac.  Two kernels, so that neither carries the other's
// gradient at the points, shared arrays and registers.
// Bound by the FP64 pipe (two FMAs a clock and SM).  What cut its work: in the passes over q
// everything that depends on u alone is a double; in 3D the projections, and the interpolation
// where its rounding is free, go one direction at a time.  A warp takes 32 volume points or 32
// face points, whichever comes next in one list, so that in small elements the two run side by
// side.  3D p = 3, 4,096 elements: residual 4.7 -> 1.3 ms, Jacobians with their right-hand
// sides 11.9 -> 7.2 ms (mixed forms 8.4); 2D p = 2, 64 elements: residual 28 -> 20 us.

// One-direction-at-a-time interpolation of F nodal fields to the volume points (3D):
// field(a, f) at the nodes -> S1 (x) -> S2 (y); the z sums are left to the point's thread.
// Fields are fastest, their stride FS odd: conflict-free both over f and over the points.
template <class Field>
__device__ __forceinline__ void interpolate_xy(const Dims& dm, const RefTables& ref, int F, int FS, double* S1,
                                               double* S2, Field field) {
  const int np1 = dm.np1, nq1 = dm.nq1;
  for (int idx = threadIdx.x; idx < F * nq1 * np1 * np1; idx += blockDim.x) {
    const int f = idx % F, t = idx / F, gx = t % nq1, ayz = t / nq1;
    double s = 0.0;
    for (int ax = 0; ax < np1; ++ax) s = fma(ref.L1[gx * np1 + ax], field(ax + np1 * ayz, f), s);
    S1[t * FS + f] = s;
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < F * nq1 * nq1 * np1; idx += blockDim.x) {
    const int f = idx % F, t = idx / F, gx = t % nq1, gy = (t / nq1) % nq1, az = t / (nq1 * nq1);
    double s = 0.0;
    for (int ay = 0; ay < np1; ++ay)
      s = fma(ref.L1[gy * np1 + ay], S1[(gx + nq1 * (ay + np1 * az)) * FS + f], s);
    S2[t * FS + f] = s;
  }
  __syncthreads();
}

// u, q at volume point g: from S2, or (null) by the dense sum over the nodes
template <int D>
__device__ __forceinline__ void volume_state(const Dims& dm, const RefTables& ref, int g, const double* su,
                                             const double* sq, const double* S2, int FS, double* u,
                                             double (*q)[D]) {
  constexpr int M = D + 2;
#pragma unroll
  for (int i = 0; i < M; ++i) {
    u[i] = 0;
#pragma unroll
    for (int j = 0; j < D; ++j) q[i][j] = 0;
  }
  if (D == 3 && S2) {
    const int np1 = dm.np1, nq2 = dm.nq1 * dm.nq1, gxy = g % nq2, gz = g / nq2;
    for (int az = 0; az < np1; ++az) {
      const double l = ref.L1[gz * np1 + az];
      const double* src = S2 + (size_t)(gxy + nq2 * az) * FS;
#pragma unroll
      for (int i = 0; i < M; ++i) {
        u[i] = fma(l, src[i], u[i]);
#pragma unroll
        for (int j = 0; j < D; ++j) q[i][j] = fma(l, src[M + i * D + j], q[i][j]);
      }
    }
    return;
  }
  const double* phi = ref.Phi + (size_t)g * dm.Np;
  for (int a = 0; a < dm.Np; ++a) {
    const double ph_a = phi[a];
#pragma unroll
    for (int i = 0; i < M; ++i) {
      u[i] += ph_a * su[a * M + i];
#pragma unroll
      for (int j = 0; j < D; ++j) q[i][j] += ph_a * sq[(a * M + i) * D + j];
    }
  }
}

// u, q and the trace state uh at face point fp
template <int D>
__device__ __forceinline__ void face_state(const Dims& dm, const RefTables& ref, const TraceTab& tt, int64_t e,
                                           int fp, const double* su, const double* sq, const double* suh,
                                           double* u, double (*q)[D], double* uh) {
  constexpr int M = D + 2;
  const int f = fp / dm.Nfq;
#pragma unroll
  for (int i = 0; i < M; ++i) {
    u[i] = 0; uh[i] = 0;
#pragma unroll
    for (int j = 0; j < D; ++j) q[i][j] = 0;
  }
  const double* phi = ref.PhiF + (size_t)fp * dm.Np;
  for (int t = 0; t < dm.Nfn; ++t) {
    const int a = ref.fnode[f * dm.Nfn + t];
    const double ph_a = phi[a];
#pragma unroll
    for (int i = 0; i < M; ++i) {
      u[i] += ph_a * su[a * M + i];
      if (!tt.nfs) uh[i] += ph_a * suh[ref.slot[a] * M + i];
#pragma unroll
      for (int j = 0; j < D; ++j) q[i][j] += ph_a * sq[(a * M + i) * D + j];
    }
  }
  if (tt.nfs) {
    // trace basis of this face from the element's table
    const int cnt = tt.nfs[e * dm.nf + f];
    const int* fsf = tt.fs + ((size_t)e * dm.nf + f) * tt.NFS;
    const double* mu = tt.muf + (((size_t)e * dm.nf + f) * dm.Nfq + (fp - f * dm.Nfq)) * tt.NFS;
    for (int j = 0; j < cnt; ++j)
#pragma unroll
      for (int i = 0; i < M; ++i) uh[i] += mu[j] * suh[fsf[j] * M + i];
  }
}

// nodal u, q and the trace nodes of element e into shared memory
__device__ __forceinline__ void load_nodal(const Dims& dm, const TraceTab& tt, const int64_t* etrace, int64_t e,
                                           const double* U, const double* Q, const double* UH, double* su,
                                           double* sq, double* suh) {
  const int m = dm.m, nu = dm.Np * m, nq = nu * dm.d;
  const int nbe = tt.nb ? tt.nb[e] : dm.Nb;
  for (int i = threadIdx.x; i < nbe * m; i += blockDim.x) suh[i] = UH[etrace[e * dm.Nb + i / m] * m + i % m];
  for (int i = threadIdx.x; i < nu; i += blockDim.x) su[i] = U[e * nu + i];
  for (int i = threadIdx.x; i < nq; i += blockDim.x) sq[i] = Q[e * nq + i];
}

template <int D, int STAB>
__global__ void k_point_jac(Dims dm, Phys ph, RefTables ref, Geo G, PointJac PJ,
                            const int64_t* __restrict__ etrace, const double* __restrict__ U,
                            const double* __restrict__ Q, const double* __restrict__ UH, TraceTab tt, int FS) {
  constexpr int M = D + 2;
  extern __shared__ double sm[];
  const int64_t e = blockIdx.x;
  const int Np = dm.Np, Nq = dm.Nq, Nfp = dm.Nfp, Nfq = dm.Nfq;
  double* su = sm;                         // [Np][M]
  double* sq = su + Np * M;                // [Np][M][D]
  double* suh = sq + Np * M * D;           // [Nb][M]
  double* S2 = FS ? suh + dm.Nb * M : nullptr;
  load_nodal(dm, tt, etrace, e, U, Q, UH, su, sq, suh);
  __syncthreads();
  if (D == 3 && FS)
    interpolate_xy(dm, ref, M * (1 + D), FS, S2 + dm.nq1 * dm.nq1 * dm.np1 * FS, S2,
                   [&](int a, int f) { return f < M ? su[a * M + f] : sq[a * M * D + f - M]; });
  const size_t jvs = (size_t)(1 + D) * D * Nq;    // stride of one (i,k) pair in Jv
  const size_t jfs = (size_t)(1 + D) * Nfp;
  const int lane = threadIdx.x & 31, nvw = (Nq + 31) / 32, nw = nvw + (Nfp + 31) / 32;
  const int wpb = blockDim.x >> 5;                // blockIdx.y: a share of the list
  for (int w32 = blockIdx.y * wpb + (threadIdx.x >> 5); w32 < nw; w32 += gridDim.y * wpb) {
  // ---- volume points
  const int g = w32 * 32 + lane, fp = g - nvw * 32;
  if (w32 < nvw && g < Nq) {
    double u[M], q[M][D];
    volume_state<D>(dm, ref, g, su, sq, S2, FS, u, q);
    const double w = G.wdet[e * Nq + g];
    double Ji[D][D];
#pragma unroll
    for (int r = 0; r < D; ++r)
#pragma unroll
      for (int j = 0; j < D; ++j) Ji[r][j] = G.Jinv[((e * Nq + g) * D + r) * D + j];
    double* jv = PJ.Jv + (size_t)e * M * M * jvs;
    float* jv32 = PJ.Jv32 ? PJ.Jv32 + (size_t)e * M * M * jvs : nullptr;
    // entry c of pair (i, k): -w sum_j Ji[r][j] dF_ij/d(unknown), c = r for u, D + l D + r for q_l
    auto put = [&](int c0, const Dual<M> (*Fd)[D]) {
#pragma unroll
      for (int i = 0; i < M; ++i)
#pragma unroll
        for (int k = 0; k < M; ++k) {
          double* o = jv + (size_t)(i * M + k) * jvs;
#pragma unroll
          for (int r = 0; r < D; ++r) {
            double s = 0;
#pragma unroll
            for (int j = 0; j < D; ++j) s += Ji[r][j] * Fd[i][j].t[k];
            o[(size_t)(c0 + r) * Nq + g] = -w * s;
            if (jv32) jv32[(size_t)(i * M + k) * jvs + (size_t)(c0 + r) * Nq + g] = (float)(-w * s);
          }
        }
    };
    flux_jacobians<D>(u, q, ph, [&](const Dual<M> (*Fd)[D]) { put(0, Fd); },
                      [&](int l, const Dual<M> (*Fd)[D]) { put(D + l * D, Fd); });
  }
  // ---- face points
  if (w32 >= nvw && fp < Nfp) {
    double u[M], uh[M], q[M][D];
    face_state<D>(dm, ref, tt, e, fp, su, sq, suh, u, q, uh);
    const double wf = G.fw[e * Nfp + fp];
    double n[D];
#pragma unroll
    for (int j = 0; j < D; ++j) n[j] = G.fn[(e * Nfp + fp) * D + j];
    double lam = 0.0;
    if constexpr (STAB == 0) lam = lf_lambda<D, double>(uh, n, ph);
    Dual<M> ud[M];
#pragma unroll
    for (int k = 0; k < M; ++k) { ud[k] = mkconst<M>(uh[k]); ud[k].t[k] = 1.0; }
    // d/duhat of the stabilisation term: LF  dlambda/duhat (u - uh) - lambda I;
    // Roe  d/duhat [ |A_n(uh)| (u - uh) ] by duals (includes - |A_n|)
    Dual<M> lamd = mkconst<M>(0.0);
    Dual<M> gd[M];
    if constexpr (STAB == 1) {
      Dual<M> dd[M];
#pragma unroll
      for (int i = 0; i < M; ++i) dd[i] = mkconst<M>(u[i]) - ud[i];
      roe_apply<D, Dual<M>>(ud, dd, n, ph, gd);
      // dfhat/du = S: its columns S e_k
#pragma unroll 1
      for (int k = 0; k < M; ++k) {
        double ek[M], sk[M];
#pragma unroll
        for (int i = 0; i < M; ++i) ek[i] = (i == k) ? 1.0 : 0.0;
        roe_apply<D, double>(uh, ek, n, ph, sk);
#pragma unroll
        for (int i = 0; i < M; ++i) {
          const size_t o = ((size_t)(e * M + i) * M + k) * Nfp + fp;
          PJ.Su[o] = wf * sk[i];
          if (PJ.Su32) PJ.Su32[o] = (float)(wf * sk[i]);
        }
      }
    } else {
      lamd = lf_lambda<D, Dual<M>>(ud, n, ph);
    }
    double* jf = PJ.Jf + (size_t)e * M * M * jfs;
    float* jf32 = PJ.Jf32 ? PJ.Jf32 + (size_t)e * M * M * jfs : nullptr;
    // entry 0 of pair (i, k): the stabilisation's derivative + dfhat/du n; entry 1 + l:
    // dfhat/dq_l n
    flux_jacobians<D>(
        uh, q, ph,
        [&](const Dual<M> (*Fd)[D]) {
#pragma unroll
          for (int i = 0; i < M; ++i)
#pragma unroll
            for (int k = 0; k < M; ++k) {
              double s = STAB == 1 ? gd[i].t[k] : lamd.t[k] * (u[i] - uh[i]) - (i == k ? lam : 0.0);
#pragma unroll
              for (int j = 0; j < D; ++j) s += Fd[i][j].t[k] * n[j];
              jf[(size_t)(i * M + k) * jfs + fp] = wf * s;
              if (jf32) jf32[(size_t)(i * M + k) * jfs + fp] = (float)(wf * s);
            }
        },
        [&](int l, const Dual<M> (*Fd)[D]) {
#pragma unroll
          for (int i = 0; i < M; ++i)
#pragma unroll
            for (int k = 0; k < M; ++k) {
              double t = 0;
#pragma unroll
              for (int j = 0; j < D; ++j) t += Fd[i][j].t[k] * n[j];
              jf[(size_t)(i * M + k) * jfs + (size_t)(1 + l) * Nfp + fp] = wf * t;
              if (jf32) jf32[(size_t)(i * M + k) * jfs + (size_t)(1 + l) * Nfp + fp] = (float)(wf * t);
            }
        });
    PJ.lamw[e * Nfp + fp] = wf * lam;
    if (PJ.lamw32) PJ.lamw32[e * Nfp + fp] = (float)(wf * lam);
    const int fk = tt.fkind ? tt.fkind[e * dm.nf + fp / Nfq] : kFaceInterior;
    if (fk != kFaceInterior) {
      double bval[M];
      boundary_point<D, STAB>(fk, uh, u, n, wf, ph, 0.0, true, PJ, e, fp, Nfp, bval);
    }
  }
  }
}

template <int D, int STAB>
__global__ void k_point_res(Dims dm, Phys ph, RefTables ref, Geo G, PointJac PJ,
                            const int64_t* __restrict__ etrace, const double* __restrict__ U,
                            const double* __restrict__ Q, const double* __restrict__ UH,
                            const double* __restrict__ UREF, double* __restrict__ RU, double* __restrict__ RHAT,
                            double* __restrict__ RHS, int64_t rhs_es, int64_t rhs_rs, TraceTab tt, int FS,
                            int work) {
  constexpr int M = D + 2;
  const bool jac = RHS != nullptr;
  extern __shared__ double sm[];
  const int64_t e = blockIdx.x;
  const int tid = threadIdx.x, nth = blockDim.x;
  const int Np = dm.Np, Nq = dm.Nq, Nb = dm.Nb, Nfp = dm.Nfp, Nfq = dm.Nfq;
  const bool has_ref = UREF != nullptr && ph.alpha != 0.0;
  double* su = sm;                         // [Np][M]
  double* sq = su + Np * M;                // [Np][M][D]
  double* suh = sq + Np * M * D;           // [Nb][M]
  double* sdu = suh + Nb * M;              // [Np][M]  u - u_ref (only with a reference state)
  double* S2 = sdu + (has_ref ? Np * M : 0);   // 3D: fields after two directions
  double* fvol = su + work;                // [M][D][Nq]  (S1 before)
  double* fsur = fvol + M * D * Nq;        // [M][Nfp]
  double* mvol = fsur + M * Nfp;           // [M][Nq]   (only with a reference state)
  double* ftr = mvol + (has_ref ? M * Nq : 0); // [M][Nfp]  flux of the trace rows (bhat on boundary faces; mixed orders)
  load_nodal(dm, tt, etrace, e, U, Q, UH, su, sq, suh);
  if (has_ref)
    for (int i = tid; i < Np * M; i += nth) sdu[i] = U[e * Np * M + i] - UREF[e * Np * M + i];
  const int nbe = tt.nb ? tt.nb[e] : Nb;         // trace slots of this element
  __syncthreads();
  if constexpr (D == 3)
    interpolate_xy(dm, ref, M * (has_ref ? 2 + D : 1 + D), FS, fvol, S2, [&](int a, int f) {
      return f < M ? su[a * M + f] : (f < M * (1 + D) ? sq[a * M * D + f - M] : sdu[a * M + f - M * (1 + D)]);
    });
  const int lane = tid & 31, nvw = (Nq + 31) / 32, nw = nvw + (Nfp + 31) / 32;
  for (int w32 = tid >> 5; w32 < nw; w32 += nth >> 5) {
  // ---- volume points
  const int g = w32 * 32 + lane, fp = g - nvw * 32;
  if (w32 < nvw && g < Nq) {
    double u[M], q[M][D];
    volume_state<D>(dm, ref, g, su, sq, D == 3 ? S2 : nullptr, FS, u, q);
    const double w = G.wdet[e * Nq + g];
    if (has_ref) {
      double du[M];
#pragma unroll
      for (int i = 0; i < M; ++i) du[i] = 0;
      if constexpr (D == 3) {
        const int np1 = dm.np1, nq2 = dm.nq1 * dm.nq1, gxy = g % nq2, gz = g / nq2;
        for (int az = 0; az < np1; ++az)
#pragma unroll
          for (int i = 0; i < M; ++i)
            du[i] = fma(ref.L1[gz * np1 + az], S2[(size_t)(gxy + nq2 * az) * FS + M * (1 + D) + i], du[i]);
      } else {
        for (int a = 0; a < Np; ++a)
#pragma unroll
          for (int i = 0; i < M; ++i) du[i] += ref.Phi[(size_t)g * Np + a] * sdu[a * M + i];
      }
#pragma unroll
      for (int i = 0; i < M; ++i) mvol[i * Nq + g] = ph.alpha * w * du[i];
    }
    double Ji[D][D];
#pragma unroll
    for (int r = 0; r < D; ++r)
#pragma unroll
      for (int j = 0; j < D; ++j) Ji[r][j] = G.Jinv[((e * Nq + g) * D + r) * D + j];
    double F[M][D];
    ns_flux<D, double, double>(u, q, ph, F);
#pragma unroll
    for (int i = 0; i < M; ++i)
#pragma unroll
      for (int r = 0; r < D; ++r) {
        double s = 0;
#pragma unroll
        for (int j = 0; j < D; ++j) s += Ji[r][j] * F[i][j];
        fvol[(i * D + r) * Nq + g] = -w * s;
      }
  }
  // ---- face points
  if (w32 >= nvw && fp < Nfp) {
    double u[M], uh[M], q[M][D];
    face_state<D>(dm, ref, tt, e, fp, su, sq, suh, u, q, uh);
    const double wf = G.fw[e * Nfp + fp];
    double n[D];
#pragma unroll
    for (int j = 0; j < D; ++j) n[j] = G.fn[(e * Nfp + fp) * D + j];
    double F[M][D];
    ns_flux<D, double, double>(uh, q, ph, F);
    // stabilisation S (u - uh): lambda I (Lax-Friedrichs) or |A_n(uh)| (Roe-type)
    double stab[M];
    double lam = 0.0;
    if constexpr (STAB == 1) {
      double dd[M];
#pragma unroll
      for (int i = 0; i < M; ++i) dd[i] = u[i] - uh[i];
      roe_apply<D, double>(uh, dd, n, ph, stab);
    } else {
      lam = lf_lambda<D, double>(uh, n, ph);
#pragma unroll
      for (int i = 0; i < M; ++i) stab[i] = lam * (u[i] - uh[i]);
    }
#pragma unroll
    for (int i = 0; i < M; ++i) {
      double s = stab[i];
#pragma unroll
      for (int j = 0; j < D; ++j) s += F[i][j] * n[j];
      fsur[i * Nfp + fp] = wf * s;
    }
    if (!tt.nfs) continue;                 // uniform order: the trace rows take fsur
    // trace rows: fhat on interior faces, the boundary flux on domain-boundary faces
    const int fk = tt.fkind ? tt.fkind[e * dm.nf + fp / Nfq] : kFaceInterior;
    if (fk != kFaceInterior) {
      double bval[M];
      boundary_point<D, STAB>(fk, uh, u, n, wf, ph, fsur[(M - 1) * Nfp + fp] / wf, false, PJ, e, fp, Nfp, bval);
#pragma unroll
      for (int i = 0; i < M; ++i) ftr[i * Nfp + fp] = bval[i];
    } else {
#pragma unroll
      for (int i = 0; i < M; ++i) ftr[i * Nfp + fp] = fsur[i * Nfp + fp];
    }
  }
  }
  __syncthreads();
  // ---- projections onto the test functions
  const double sgn = jac ? -1.0 : 1.0;
  // right-hand side column: uniform meshes e * rhs_es, row stride rhs_rs; meshes with
  // per-element sizes: column n_e of the element's bordered matrix
  double* rhs_e = nullptr;
  int64_t rrs = rhs_rs;
  if (jac) {
    if (tt.soff && rhs_rs != 1) {
      rhs_e = RHS + tt.soff[e] + dm.nu + (int64_t)M * nbe;
      rrs = tt.ldv[e];
    } else {
      rhs_e = RHS + e * rhs_es;
    }
  }
  if constexpr (D == 3) {
    // one direction at a time (z, y, x; the time term joins direction 2, whose y and x
    // stages are L (x) L), faces in two 1D stages; the nodal arrays are free now
    const int np1 = dm.np1, nq1 = dm.nq1, TS = nq1 * nq1 * np1, VS = nq1 * np1 * np1, FB = nq1 * np1, Nfn1 = np1 * np1;
    double* t1 = su;                       // [M][3][TS]
    double* t2 = t1 + M * 3 * TS;          // [M][2][VS]
    double* fu = t2 + M * 2 * VS;          // [M][6][FB]
    double* fb = fu + M * 6 * FB;          // [M][6][Nfn]
    const double *L = ref.L1, *dL = ref.dL1;
    for (int idx = tid; idx < M * 6 * FB; idx += nth) {
      const int i = idx / (6 * FB), f = (idx / FB) % 6, t = idx % FB, a0 = t % np1, g1 = t / np1;
      const double* src = fsur + i * Nfp + f * Nfq + nq1 * g1;
      double s = 0.0;
      for (int g0 = 0; g0 < nq1; ++g0) s = fma(L[g0 * np1 + a0], src[g0], s);
      fu[idx] = s;
    }
    for (int idx = tid; idx < M * 3 * TS; idx += nth) {
      const int i = idx / (3 * TS), r = (idx / TS) % 3, t = idx % TS, gxy = t % (nq1 * nq1), az = t / (nq1 * nq1);
      const double* X = r == 2 ? dL : L;
      const double* src = fvol + (i * D + r) * Nq + gxy;
      double s = 0.0;
      for (int gz = 0; gz < nq1; ++gz) s = fma(X[gz * np1 + az], src[nq1 * nq1 * gz], s);
      if (r == 2 && has_ref) {
        const double* ms = mvol + i * Nq + gxy;
        for (int gz = 0; gz < nq1; ++gz) s = fma(L[gz * np1 + az], ms[nq1 * nq1 * gz], s);
      }
      t1[idx] = s;
    }
    __syncthreads();
    for (int idx = tid; idx < M * VS; idx += nth) {
      const int i = idx / VS, t = idx % VS, gx = t % nq1, ay = (t / nq1) % np1, az = t / (nq1 * np1);
      const double *T0 = t1 + i * 3 * TS, *T1 = T0 + TS, *T2 = T1 + TS;
      double s0 = 0.0, s1 = 0.0;
      for (int gy = 0; gy < nq1; ++gy) {
        const int q = gx + nq1 * (gy + nq1 * az);
        s0 = fma(L[gy * np1 + ay], T0[q], s0);
        s1 = fma(dL[gy * np1 + ay], T1[q], s1);
        s1 = fma(L[gy * np1 + ay], T2[q], s1);
      }
      t2[(i * 2 + 0) * VS + t] = s0;
      t2[(i * 2 + 1) * VS + t] = s1;
    }
    for (int idx = tid; idx < M * 6 * Nfn1; idx += nth) {
      const int i = idx / (6 * Nfn1), f = (idx / Nfn1) % 6, tn = idx % Nfn1, a0 = tn % np1, a1 = tn / np1;
      const double* src = fu + ((size_t)i * 6 + f) * FB + a0;
      double s = 0.0;
      for (int g1 = 0; g1 < nq1; ++g1) s = fma(L[g1 * np1 + a1], src[np1 * g1], s);
      fb[idx] = s;
    }
    __syncthreads();
    for (int ai = tid; ai < Np * M; ai += nth) {
      const int a = ai / M, i = ai % M, ax = a % np1, ayz = a / np1;
      const double *V0 = t2 + i * 2 * VS + nq1 * ayz, *V1 = V0 + VS;
      double s = 0.0;
      for (int gx = 0; gx < nq1; ++gx) {
        s = fma(dL[gx * np1 + ax], V0[gx], s);
        s = fma(L[gx * np1 + ax], V1[gx], s);
      }
      if (ref.slot[a] >= 0) s += face_part(dm, fb, i, a);
      if (jac) rhs_e[((int64_t)i * Np + a) * rrs] = sgn * s;
      else if (RU) RU[(e * Np + a) * M + i] = s;
    }
    if (!tt.nfs) {                         // uniform order: a trace row is its node's face part
      for (int si = nth - 1 - tid; si < nbe * M; si += nth) {
        const int s = si / M, i = si % M;
        const double t = face_part(dm, fb, i, ref.bnode[s]);
        if (jac) rhs_e[((int64_t)dm.nu + (int64_t)i * nbe + s) * rrs] = sgn * t;
        else RHAT[(e * Nb + s) * M + i] = t;
      }
      return;
    }
  } else {
  for (int ai = tid; ai < Np * M; ai += nth) {
    const int a = ai / M, i = ai % M;
    double s = 0;
    for (int g = 0; g < Nq; ++g) {
      double t = has_ref ? ref.Phi[(size_t)g * Np + a] * mvol[i * Nq + g] : 0.0;
#pragma unroll
      for (int r = 0; r < D; ++r) t += ref.Dxi[((size_t)r * Nq + g) * Np + a] * fvol[(i * D + r) * Nq + g];
      s += t;
    }
    if (ref.slot[a] >= 0)
      for (int fp = 0; fp < Nfp; ++fp) s += ref.PhiF[(size_t)fp * Np + a] * fsur[i * Nfp + fp];
    if (jac) rhs_e[((int64_t)i * Np + a) * rrs] = sgn * s;
    else if (RU) RU[(e * Np + a) * M + i] = s;
  }
  }
  for (int si = nth - 1 - tid; si < nbe * M; si += nth) {
    const int s = si / M, i = si % M;
    double t = 0;
    if (tt.nfs) {
      const int* fl = tt.sfl + ((size_t)e * Nb + s) * 3;
      for (int c = 0; c < 3; ++c) {
        const int code = fl[c];
        if (code < 0) continue;
        const int f = code / tt.NFS, j = code % tt.NFS;
        const double* mu = tt.muf + ((size_t)e * dm.nf + f) * Nfq * tt.NFS + j;
        for (int gf = 0; gf < Nfq; ++gf) t += mu[(size_t)gf * tt.NFS] * ftr[i * Nfp + f * Nfq + gf];
      }
    } else {
      const int a = ref.bnode[s];
      for (int fp = 0; fp < Nfp; ++fp) t += ref.PhiF[(size_t)fp * Np + a] * fsur[i * Nfp + fp];
    }
    if (jac) rhs_e[((int64_t)dm.nu + (int64_t)i * nbe + s) * rrs] = sgn * t;
    else RHAT[(e * Nb + s) * M + i] = t;
  }
}

// Blocks of 128 threads that keep every SM of the current device evenly busy (8 per SM).
cudaError_t spread_blocks(int64_t* blocks) {
  int dev = 0, sms = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err == cudaSuccess) err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  *blocks = 8 * (int64_t)sms;
  return err;
}

// q*[e][c][k][l] = sum_t H_l[c][t] uhat_k(t) - sum_b G_l[c][b] u_k(b)
// One output a thread, an element's outputs over several blocks: a thread's chain of loads and
// FMAs is as long as a row, and with one block per element a mesh of few large elements left
// most of the chip idle behind it.  3D p = 4, 210 elements 0.48 -> 0.17 ms;
// 175 elements of orders 2..4 0.80 -> 0.13 ms; 4,096 at p = 3 0.79 -> 0.77 (FP64 pipe).
__global__ void k_lift(Dims dm, Geo G, const int64_t* __restrict__ etrace, const double* __restrict__ U,
                       const double* __restrict__ UH, double* __restrict__ QS, TraceTab tt) {
  extern __shared__ double sm[];
  const int64_t e = blockIdx.x;
  const int tid = threadIdx.x, nth = blockDim.x;
  const int Np = dm.Np, Nb = dm.Nb, m = dm.m, d = dm.d;
  double* su = sm;            // [Np][m]
  double* suh = su + Np * m;  // [Nb][m]
  for (int i = tid; i < Np * m; i += nth) su[i] = U[e * Np * m + i];
  const int nbe = tt.nb ? tt.nb[e] : Nb;
  for (int i = tid; i < nbe * m; i += nth) suh[i] = UH[etrace[e * Nb + i / m] * m + i % m];
  __syncthreads();
  const int idx = blockIdx.y * nth + tid;
  if (idx < Np * m * d) {
    int c = idx / (m * d), k = (idx / d) % m, l = idx % d;
    const double* gl = G.Gl + (((size_t)e * d + l) * Np + c) * Np;
    const double* hl = G.Hl + (((size_t)e * d + l) * Np + c) * Nb;
    double s = 0;
    for (int t = 0; t < nbe; ++t) s += hl[t] * suh[t * m + k];
    for (int b = 0; b < Np; ++b) s -= gl[b] * su[b * m + k];
    QS[e * Np * m * d + idx] = s;
  }
}

// R_q = M (q - q*), optionally rhoq = q - q*; small meshes over several blocks per element
// (3D p = 4, 210 elements, both forms together 0.21 -> 0.12 ms).
__global__ void k_rq(Dims dm, Geo G, const double* __restrict__ Q, const double* __restrict__ QS,
                     double* __restrict__ RQ, double* __restrict__ RHOQ) {
  extern __shared__ double sm[];
  const int64_t e = blockIdx.x;
  const int tid = threadIdx.x, nth = blockDim.x;
  const int Np = dm.Np, w = dm.m * dm.d;
  double* dq = sm;   // [Np][m d]
  for (int i = tid; i < Np * w; i += nth) {
    double v = Q[e * Np * w + i] - QS[e * Np * w + i];
    dq[i] = v;
    if (RHOQ && blockIdx.y == 0) RHOQ[e * Np * w + i] = v;
  }
  __syncthreads();
  if (!RQ) return;
  const double* Ms = G.Mass + (size_t)e * Np * Np;
  for (int idx = blockIdx.y * nth + tid; idx < Np * w; idx += nth * gridDim.y) {
    int a = idx / w, c = idx % w;
    double s = 0;
    for (int b = 0; b < Np; ++b) s += Ms[a * Np + b] * dq[b * w + c];
    RQ[e * Np * w + idx] = s;
  }
}

}  // namespace

cudaError_t launch_points(iedg_mesh* M, const double* u, const double* q, const double* qs,
                          const double* uhat, const double* u_ref, bool jacobians, double* r_u,
                          double* rhat, cudaStream_t st) {
  const Dims& dm = M->dm;
  const int threads = 128;
  const size_t nodal = (size_t)dm.Np * dm.m * (1 + dm.d) + (size_t)dm.Nb * dm.m;
  const size_t np1 = dm.np1, nq1 = dm.nq1;
  cudaError_t err;
  if (jacobians) {
    // mixed forms: K depends on the FP32 roundings of these Jacobians, so u and q at the
    // points keep the order of the dense sum; FP64 forms in 3D sum one direction at a time
    const int FS = dm.d == 3 && M->precision == 0 ? (dm.m * (1 + dm.d)) | 1 : 0;
    const size_t smem = sizeof(double) * (nodal + FS * (nq1 * nq1 * np1 + nq1 * np1 * np1));
    auto kern = dm.d == 2 ? (M->ph.stab == 1 ? k_point_jac<2, 1> : k_point_jac<2, 0>)
                          : (M->ph.stab == 1 ? k_point_jac<3, 1> : k_point_jac<3, 0>);
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    // An element's warps over several blocks where the elements alone are too few to fill the
    // chip evenly (below spread_blocks): each block repeats the nodal loads (and, in FP64, the
    // interpolation), which large meshes need not pay.  3D p = 4, 210 elements 1.0 -> 0.84 ms
    // (FP32 1.34 -> 1.10); 175 elements of orders 2..4 1.9 -> 1.2 ms.
    const int items = (dm.Nq + 31) / 32 + (dm.Nfp + 31) / 32, most = (items + threads / 32 - 1) / (threads / 32);
    int64_t spread = 0;
    err = spread_blocks(&spread);
    if (err != cudaSuccess) return err;
    const int64_t want = (spread + M->E - 1) / M->E;
    const dim3 grid((unsigned)M->E, (unsigned)(want < most ? want : most));
    kern<<<grid, threads, smem, st>>>(dm, M->ph, M->ref, M->geo, M->pj, M->etrace, u, q, uhat, M->tt, FS);
    err = cudaGetLastError();
    if (err != cudaSuccess) return err;
  }
  const bool has_ref = u_ref && M->ph.alpha != 0.0;
  const int FS = dm.d == 3 ? (dm.m * (1 + dm.d + (has_ref ? 1 : 0))) | 1 : 0;
  // nodal arrays and S2, later (3D) the projection stages; S1, later the fluxes at the points
  size_t work = nodal + (has_ref ? (size_t)dm.Np * dm.m : 0) + FS * nq1 * nq1 * np1;
  size_t points = (size_t)dm.m * dm.d * dm.Nq + (has_ref ? dm.m * dm.Nq : 0) +
                  (size_t)(M->tt.nfs ? 2 : 1) * dm.m * dm.Nfp;
  if (dm.d == 3) {
    const size_t stages = dm.m * (3 * nq1 * nq1 * np1 + 2 * nq1 * np1 * np1 + 6 * nq1 * np1 + 6 * np1 * np1);
    work = work > stages ? work : stages;
    points = points > FS * nq1 * np1 * np1 ? points : FS * nq1 * np1 * np1;
  }
  const size_t smem = sizeof(double) * (work + points);
  // right-hand sides: column n of the FP64 bordered matrix, or the FP64 rhs array
  // (ragged FP64 matrices: the kernel adds the element's offset and n_e to S itself)
  double* rhs = !jacobians ? nullptr : (M->precision == 0 ? (M->tt.soff ? M->S : M->S + dm.n) : M->rhs64);
  int64_t es = M->precision == 0 ? (int64_t)dm.n * dm.ld : dm.n;
  int64_t rs = M->precision == 0 ? dm.ld : 1;
  auto kern = dm.d == 2 ? (M->ph.stab == 1 ? k_point_res<2, 1> : k_point_res<2, 0>)
                        : (M->ph.stab == 1 ? k_point_res<3, 1> : k_point_res<3, 0>);
  err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  kern<<<(unsigned)M->E, threads, smem, st>>>(dm, M->ph, M->ref, M->geo, M->pj, M->etrace, u, jacobians ? qs : q,
                                              uhat, u_ref, r_u, rhat, rhs, es, rs, M->tt, FS, (int)work);
  return cudaGetLastError();
}

cudaError_t launch_lift(iedg_mesh* M, const double* u, const double* uhat, double* qstar, cudaStream_t st) {
  const Dims& dm = M->dm;
  size_t smem = sizeof(double) * (size_t)(dm.Np + dm.Nb) * dm.m;
  const dim3 grid((unsigned)M->E, (unsigned)idiv_up(dm.Np * dm.m * dm.d, 128));
  k_lift<<<grid, 128, smem, st>>>(dm, M->geo, M->etrace, u, uhat, qstar, M->tt);
  return cudaGetLastError();
}

cudaError_t launch_rq(iedg_mesh* M, const double* q, const double* qs, double* r_q, double* rhoq,
                      cudaStream_t st) {
  const Dims& dm = M->dm;
  size_t smem = sizeof(double) * (size_t)dm.Np * dm.m * dm.d;
  int64_t spread = 0;
  const cudaError_t err = spread_blocks(&spread);
  if (err != cudaSuccess) return err;
  const int64_t want = (spread + M->E - 1) / M->E, most = idiv_up(dm.Np * dm.m * dm.d, 128);
  const dim3 grid((unsigned)M->E, r_q ? (unsigned)(want < most ? want : most) : 1u);
  k_rq<<<grid, 128, smem, st>>>(dm, M->geo, q, qs, r_q, rhoq);
  return cudaGetLastError();
}

}  // namespace iedg
