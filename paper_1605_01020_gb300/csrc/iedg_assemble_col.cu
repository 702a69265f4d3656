// Element block assembly with one thread per column of an (i, k) block (uniform meshes,
// p + 2 points per direction): small elements (2D of degree 1..3, 3D of degree 1; FP64 and
// FP32) and, in FP32, hexahedra of degree 2..4.
//
// Same element matrix as k_assemble (iedg_assemble.cu).  A column of a small element
// fits in registers, so a thread forms its right operand point by point, contracts it
// with the test functions as it goes and writes its rows; nothing is exchanged between
// threads and there is no barrier.  k_assemble gives an (i, k) block of a small element
// to 256 threads of which its 4 x 8 tiles keep few busy (16 at 2D p = 3), with eight
// barriers a block.
// FP64: the contraction is sum-factorised (x, then y, then z), which halves the
// multiply-adds of the FP64 pipe, the bound.  FP32 (mixed path): the dense contraction
// in k_assemble's order, so the FP32 element matrix stays the same bit for bit.
// Measured, FP64, k_assemble -> this kernel: 2D p = 3, 851 elements 4.32 -> 0.54 ms;
// 2D p = 2, 64 elements 213 -> 26 us.
#include "iedg_internal.cuh"

namespace iedg {
namespace {

constexpr int AC_THREADS = 128;

template <int NP1>
__host__ __device__ constexpr int ipow(int d) { return d == 0 ? 1 : NP1 * ipow<NP1>(d - 1); }

// a b rounded: keeps the compiler from contracting it into a following addition, so that
// the FP32 form rounds where k_assemble's loops do
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return a * b; }

template <class T, int D, int NP1, int NQ1>
__global__ void __launch_bounds__(AC_THREADS)
k_assemble_col(Dims dm, Phys ph, RefTables ref, AsmTab<T> tb, T* __restrict__ S, const double* __restrict__ rhs64,
               int64_t E) {
  constexpr int m = D + 2, m2 = m * m, Np = ipow<NP1>(D), Nq = ipow<NQ1>(D), Nfq = ipow<NQ1>(D - 1);
  constexpr int Nfn = ipow<NP1>(D - 1), nf = 2 * D, Nfp = nf * Nfq;
  constexpr int Nb = Np - (NP1 > 2 ? ipow<(NP1 > 2 ? NP1 - 2 : 1)>(D) : 0), ncol = Np + Nb;
  __shared__ T sL[NQ1][NP1], sD[NQ1][NP1];
  __shared__ int sbn[Nb];
  for (int i = threadIdx.x; i < NQ1 * NP1; i += AC_THREADS) {
    sL[i / NP1][i % NP1] = (T)ref.L1[i];
    sD[i / NP1][i % NP1] = (T)ref.dL1[i];
  }
  for (int i = threadIdx.x; i < Nb; i += AC_THREADS) sbn[i] = ref.bnode[i];
  __syncthreads();
  const int64_t idx = (int64_t)blockIdx.x * AC_THREADS + threadIdx.x;
  if (idx >= E * m2 * ncol) return;
  const int64_t e = idx / (m2 * ncol);
  const int rem = (int)(idx % (m2 * ncol)), pair = rem / ncol, col = rem % ncol, i = pair / m, k = pair % m;
  const bool ucol = col < Np;
  const int t = col - Np;
  // u-columns take -G_l and the basis value, trace columns +H_l and the trace basis
  const T* GV = ucol ? tb.GlV + (size_t)e * D * Nq * Np + col : tb.HlV + (size_t)e * D * Nq * Nb + t;
  const T* GF = ucol ? tb.GlF + (size_t)e * D * Nfp * Np + col : tb.HlF + (size_t)e * D * Nfp * Nb + t;
  const int st = ucol ? Np : Nb, bcol = ucol ? col : sbn[t];
  const T sg = ucol ? (T)-1 : (T)1;
  const T* jv = tb.Jv + ((size_t)e * m2 + pair) * (size_t)((1 + D) * D * Nq);
  const T* jf = tb.Jf + ((size_t)e * m2 + pair) * (size_t)((1 + D) * Nfp);
  // right operand of reference direction r at volume point g
  auto wvol = [&](int g, T (&w)[D]) {
    const T phi = ucol ? tb.Phi[(size_t)g * Np + col] : (T)0;
    T gl[D];
#pragma unroll
    for (int l = 0; l < D; ++l) gl[l] = sg * GV[((size_t)l * Nq + g) * st];
#pragma unroll
    for (int r = 0; r < D; ++r) {
      T v = mul(jv[(size_t)r * Nq + g], phi);
#pragma unroll
      for (int l = 0; l < D; ++l) v = fma(jv[(size_t)(D + l * D + r) * Nq + g], gl[l], v);
      w[r] = v;
    }
  };
  T acc[Np];
#pragma unroll
  for (int a = 0; a < Np; ++a) acc[a] = (T)0;
  if constexpr (sizeof(T) == 8) {
    constexpr int PL = NP1 * NP1, NZ = D == 3 ? NQ1 : 1;
#pragma unroll 1
    for (int gz = 0; gz < NZ; ++gz) {
      T p01[PL], p2[PL];       // D = 3: the plane's L and L' (z) operands; D = 2: p01 is the result
#pragma unroll
      for (int a = 0; a < PL; ++a) p01[a] = p2[a] = (T)0;
#pragma unroll
      for (int gy = 0; gy < NQ1; ++gy) {
        T s[D][NP1];
#pragma unroll
        for (int r = 0; r < D; ++r)
#pragma unroll
          for (int a = 0; a < NP1; ++a) s[r][a] = (T)0;
#pragma unroll
        for (int gx = 0; gx < NQ1; ++gx) {
          T w[D];
          wvol(gx + NQ1 * (gy + NQ1 * gz), w);
#pragma unroll
          for (int a = 0; a < NP1; ++a) {
            s[0][a] = fma(sD[gx][a], w[0], s[0][a]);
#pragma unroll
            for (int r = 1; r < D; ++r) s[r][a] = fma(sL[gx][a], w[r], s[r][a]);
          }
        }
#pragma unroll
        for (int ay = 0; ay < NP1; ++ay)
#pragma unroll
          for (int ax = 0; ax < NP1; ++ax) {
            p01[ay * NP1 + ax] = fma(sD[gy][ay], s[1][ax], fma(sL[gy][ay], s[0][ax], p01[ay * NP1 + ax]));
            if constexpr (D == 3) p2[ay * NP1 + ax] = fma(sL[gy][ay], s[D - 1][ax], p2[ay * NP1 + ax]);
          }
      }
      if constexpr (D == 2) {
#pragma unroll
        for (int a = 0; a < PL; ++a) acc[a] = p01[a];
      } else {
#pragma unroll
        for (int az = 0; az < NP1; ++az)
#pragma unroll
          for (int a = 0; a < PL; ++a)
            acc[az * PL + a] = fma(sD[gz][az], p2[a], fma(sL[gz][az], p01[a], acc[az * PL + a]));
      }
    }
  } else {
#pragma unroll 1
    for (int g = 0; g < Nq; ++g) {
      T w[D];
      wvol(g, w);
#pragma unroll
      for (int r = 0; r < D; ++r)
#pragma unroll
        for (int a = 0; a < Np; ++a) acc[a] = fma(tb.Dxi[((size_t)r * Nq + g) * Np + a], w[r], acc[a]);
    }
  }
  // face parts of the boundary rows
  T fac[Np];
#pragma unroll
  for (int a = 0; a < Np; ++a) fac[a] = (T)0;
#pragma unroll
  for (int f = 0; f < nf; ++f) {
    T s[Nfn];
#pragma unroll
    for (int a = 0; a < Nfn; ++a) s[a] = (T)0;
#pragma unroll
    for (int gf = 0; gf < Nfq; ++gf) {
      const int fp = f * Nfq + gf;
      // dfhat/du: lambda I (Lax-Friedrichs) or the pair's entry of S (Roe-type)
      T cf = jf[fp];
      if (ucol) cf = tb.Su ? tb.Su[((size_t)e * m2 + pair) * Nfp + fp] : (i == k ? tb.lamw[e * Nfp + fp] : (T)0);
      T v = mul(cf, tb.PhiF[(size_t)fp * Np + bcol]);
#pragma unroll
      for (int l = 0; l < D; ++l) v = fma(jf[(size_t)(1 + l) * Nfp + fp], sg * GF[((size_t)l * Nfp + fp) * st], v);
#pragma unroll
      for (int tn = 0; tn < Nfn; ++tn) {
        // face node tn: its coordinates over the face's tangential directions in order
        int a = 0, str = 1, q = tn;
#pragma unroll
        for (int dir = 0; dir < D; ++dir) {
          int c;
          if (dir == f / 2) c = (f & 1) ? NP1 - 1 : 0;
          else { c = q % NP1; q /= NP1; }
          a += c * str;
          str *= NP1;
        }
        s[tn] = fma(tb.PhiF[(size_t)fp * Np + a], v, s[tn]);
      }
    }
#pragma unroll
    for (int tn = 0; tn < Nfn; ++tn) {
      int a = 0, str = 1, q = tn;
#pragma unroll
      for (int dir = 0; dir < D; ++dir) {
        int c;
        if (dir == f / 2) c = (f & 1) ? NP1 - 1 : 0;
        else { c = q % NP1; q /= NP1; }
        a += c * str;
        str *= NP1;
      }
      fac[a] += s[tn];
    }
  }
  // write the column
  T* Se = S + e * (int64_t)dm.n * dm.ld;
  const int64_t cs = ucol ? (int64_t)k * Np + col : (int64_t)dm.nu + (int64_t)k * Nb + t;
  int sl = 0;
#pragma unroll
  for (int a = 0; a < Np; ++a) {
    bool bnd = false;
    int q = a;
#pragma unroll
    for (int dir = 0; dir < D; ++dir) { const int c = q % NP1; q /= NP1; bnd = bnd || c == 0 || c == NP1 - 1; }
    T v = acc[a];
    if (bnd) v += fac[a];
    if (i == k && ucol) v = fma((T)ph.alpha, tb.Mass[((size_t)e * Np + a) * Np + col], v);
    Se[((int64_t)i * Np + a) * dm.ld + cs] = v;
    if (bnd) {
      Se[((int64_t)dm.nu + (int64_t)i * Nb + sl) * dm.ld + cs] = fac[a];
      ++sl;
    }
  }
  if (rhs64 != nullptr && pair == 0)
    for (int r = col; r < dm.n; r += ncol) Se[(int64_t)r * dm.ld + dm.n] = (T)rhs64[e * dm.n + r];
}

// FP32 hexahedra of degree 2..4 (mixed path).  The sum-factorised contraction of
// iedg_assemble_sf.cu (z, then y, then x) needs, for the test functions of one z layer of
// a column, (p+1)^2 sums of the x stage, 2 (p+1) of the y stage and 3 of the z stage.  Two
// threads share a column, each with half of the z layers in registers (110 to 160 of
// them), so nothing goes through shared memory between barriers (nine per 16 columns
// there).  The halves sit in different warps, which makes the 1D tables, kernel
// parameters, constant operands of the multiply-adds.  A z layer's share of the faces is
// its row of the x and y faces and, at the ends, a z face.  Every value is formed by the
// same operations in the same order as there, so the FP32 element matrix is the same bit
// for bit.  Bound by load instructions and their latency (16 per point: 12 coefficients
// that a warp shares, 4 table values per lane).
// Measured, all elements, iedg_assemble_sf.cu's uniform form -> this kernel: p = 3, 4096
// elements 24.1 -> 13.6 ms; p = 4, 210 elements 8.3 -> 2.5 ms (spills: 14 warps share the
// registers); p = 3, 504 elements 3.0 -> 1.7 ms.  With coefficients read from global memory
// per point: 27.8, 5.1, 3.5 ms.  Issue slots 55 % busy at p = 3.
template <int NP1>
struct Tab1D {
  float L[NP1 + 1][NP1], D[NP1 + 1][NP1];
};

// Point coefficients of the CTA's pair.
template <int NP1>
struct HexCoef {
  float4 v[(NP1 + 1) * (NP1 + 1) * (NP1 + 1)][3];   // cu_0..2, cq_lr (l slow)
  float4 f[6 * (NP1 + 1) * (NP1 + 1)];              // fq_0..2, fuh
  float fu[6 * (NP1 + 1) * (NP1 + 1)];              // S_ik or lambda delta_ik
};

// One column's rows of the z layers Z0 .. Z0 + NZ - 1.
template <int NP1, int Z0, int NZ>
__device__ __forceinline__ void hex32_layers(const HexCoef<NP1>& cs, int i, int k, int col, bool ucol, bool cq, int64_t e,
                                             int64_t ld, float alpha, const RefTables& ref, const AsmTab<float>& tb,
                                             float* Su, float* St, const Tab1D<NP1>& tab) {
  constexpr int NQ1 = NP1 + 1, Np = NP1 * NP1 * NP1, Nq = NQ1 * NQ1 * NQ1, Nfq = NQ1 * NQ1, Nfp = 6 * Nfq;
  constexpr int Nb = Np - (NP1 - 2) * (NP1 - 2) * (NP1 - 2), PL = NP1 * NP1;
  const int st = ucol ? Np : Nb;
  const float sg = ucol ? -1.f : 1.f;
  float fac[NZ * PL];                     // face parts of the layers' nodes, az PL + ay NP1 + ax
#pragma unroll
  for (int a = 0; a < NZ * PL; ++a) fac[a] = 0.f;
  {
    // right operand at the face points, two 1D stages per face, faces summed in order
    const float* GF = ucol ? tb.GlF + (size_t)e * 3 * Nfp * Np + col : tb.HlF + (size_t)e * 3 * Nfp * Nb + col;
    const float* pf = tb.PhiF + (ucol ? col : ref.bnode[col]);
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      if ((f == 4 && Z0 > 0) || (f == 5 && Z0 + NZ < NP1)) continue;
      constexpr int NA = NP1 > NZ ? NP1 : NZ;
      const int n2 = f < 4 ? NZ : NP1, b2 = f < 4 ? Z0 : 0;     // second tangential index: z, or y on z faces
      float fn[NA * NP1];
#pragma unroll
      for (int a = 0; a < NA * NP1; ++a) fn[a] = 0.f;
#pragma unroll 1
      for (int g1 = 0; g1 < NQ1; ++g1) {
        float u[NA];
#pragma unroll
        for (int a = 0; a < NA; ++a) u[a] = 0.f;
#pragma unroll
        for (int g2 = 0; g2 < NQ1; ++g2) {
          const int fp = f * Nfq + g1 + NQ1 * g2;
          const float4 c4 = cs.f[fp];
          float v = mul(ucol ? cs.fu[fp] : c4.w, pf[(size_t)fp * Np]);
          if (cq) {
            v = fmaf(c4.x, sg * GF[(size_t)fp * st], v);
            v = fmaf(c4.y, sg * GF[((size_t)Nfp + fp) * st], v);
            v = fmaf(c4.z, sg * GF[((size_t)2 * Nfp + fp) * st], v);
          }
#pragma unroll
          for (int a = 0; a < NA; ++a)
            if (a < n2) u[a] = fmaf(tab.L[g2][b2 + a], v, u[a]);
        }
#pragma unroll
        for (int a2 = 0; a2 < NA; ++a2)
          if (a2 < n2)
#pragma unroll
            for (int a1 = 0; a1 < NP1; ++a1) fn[a2 * NP1 + a1] = fmaf(tab.L[g1][a1], u[a2], fn[a2 * NP1 + a1]);
      }
#pragma unroll
      for (int a2 = 0; a2 < NA; ++a2)
        if (a2 < n2)
#pragma unroll
          for (int a1 = 0; a1 < NP1; ++a1) {
            const int s = (f & 1) ? NP1 - 1 : 0;
            const int a = f / 2 == 0 ? a2 * PL + a1 * NP1 + s
                                     : (f / 2 == 1 ? a2 * PL + s * NP1 + a1 : (s == 0 ? 0 : NZ - 1) * PL + a2 * NP1 + a1);
            fac[a] += fn[a2 * NP1 + a1];
          }
    }
  }
  float out[NZ * PL];
#pragma unroll
  for (int a = 0; a < NZ * PL; ++a) out[a] = 0.f;
  if (ucol || cq) {
    const float* GV = ucol ? tb.GlV + (size_t)e * 3 * Nq * Np + col : tb.HlV + (size_t)e * 3 * Nq * Nb + col;
    const float* ph = tb.Phi + (ucol ? col : 0);
    // table values of a line of points in z, read one line ahead
    float nx[NQ1][4];
    auto fetch = [&](int gxy) {
#pragma unroll
      for (int gz = 0; gz < NQ1; ++gz) {
        const int g = gxy + NQ1 * NQ1 * gz;
        nx[gz][3] = ucol ? ph[(size_t)g * Np] : 0.f;
#pragma unroll
        for (int l = 0; l < 3; ++l) nx[gz][l] = cq ? GV[((size_t)l * Nq + g) * st] : 0.f;
      }
    };
    fetch(0);
#pragma unroll 1
    for (int gx = 0; gx < NQ1; ++gx) {
      float V0[NZ * NP1], V1[NZ * NP1];
#pragma unroll
      for (int a = 0; a < NZ * NP1; ++a) V0[a] = V1[a] = 0.f;
#pragma unroll 1
      for (int gy = 0; gy < NQ1; ++gy) {
        float T0[NZ], T1[NZ], T2[NZ];
#pragma unroll
        for (int a = 0; a < NZ; ++a) T0[a] = T1[a] = T2[a] = 0.f;
        float t[NQ1][4];
#pragma unroll
        for (int gz = 0; gz < NQ1; ++gz)
#pragma unroll
          for (int l = 0; l < 4; ++l) t[gz][l] = l < 3 ? sg * nx[gz][l] : nx[gz][l];
        const int next = gy + 1 < NQ1 ? gx + NQ1 * (gy + 1) : gx + 1;
        if (next < NQ1 * NQ1) fetch(next);
#pragma unroll
        for (int gz = 0; gz < NQ1; ++gz) {
          const int g = gx + NQ1 * (gy + NQ1 * gz);
          const float4 c0 = cs.v[g][0], c1 = cs.v[g][1], c2 = cs.v[g][2];
          float w[3] = {mul(c0.x, t[gz][3]), mul(c0.y, t[gz][3]), mul(c0.z, t[gz][3])};
          if (cq) {
            w[0] = fmaf(c0.w, t[gz][0], w[0]);
            w[1] = fmaf(c1.x, t[gz][0], w[1]);
            w[2] = fmaf(c1.y, t[gz][0], w[2]);
            w[0] = fmaf(c1.z, t[gz][1], w[0]);
            w[1] = fmaf(c1.w, t[gz][1], w[1]);
            w[2] = fmaf(c2.x, t[gz][1], w[2]);
            w[0] = fmaf(c2.y, t[gz][2], w[0]);
            w[1] = fmaf(c2.z, t[gz][2], w[1]);
            w[2] = fmaf(c2.w, t[gz][2], w[2]);
          }
#pragma unroll
          for (int a = 0; a < NZ; ++a) {
            T0[a] = fmaf(tab.L[gz][Z0 + a], w[0], T0[a]);
            T1[a] = fmaf(tab.L[gz][Z0 + a], w[1], T1[a]);
            T2[a] = fmaf(tab.D[gz][Z0 + a], w[2], T2[a]);
          }
        }
#pragma unroll
        for (int az = 0; az < NZ; ++az)
#pragma unroll
          for (int ay = 0; ay < NP1; ++ay) {
            const int q = az * NP1 + ay;
            V0[q] = fmaf(tab.L[gy][ay], T0[az], V0[q]);
            V1[q] = fmaf(tab.D[gy][ay], T1[az], V1[q]);
            V1[q] = fmaf(tab.L[gy][ay], T2[az], V1[q]);
          }
      }
#pragma unroll
      for (int q = 0; q < NZ * NP1; ++q)
#pragma unroll
        for (int ax = 0; ax < NP1; ++ax) {
          out[q * NP1 + ax] = fmaf(tab.D[gx][ax], V0[q], out[q * NP1 + ax]);
          out[q * NP1 + ax] = fmaf(tab.L[gx][ax], V1[q], out[q * NP1 + ax]);
        }
    }
  }
  // u-rows: volume + face part + mass; trace rows: face parts.  Slots count the boundary
  // nodes in node order: all of an end layer, the rim of an inner one.
#pragma unroll
  for (int j = 0; j < NZ * PL; ++j) {
    const int az = Z0 + j / PL, ay = (j / NP1) % NP1, ax = j % NP1, a = Z0 * PL + j;
    constexpr int RIM = 4 * (NP1 - 1);
    const bool end = az == 0 || az == NP1 - 1, rim = ax == 0 || ax == NP1 - 1 || ay == 0 || ay == NP1 - 1;
    float v = out[j];
    if (end || rim) {
      v += fac[j];
      const int in_layer = end ? ay * NP1 + ax
                               : (ay == 0 ? ax : (ay == NP1 - 1 ? NP1 + 2 * (NP1 - 2) + ax : NP1 + 2 * (ay - 1) + (ax > 0)));
      const int before = az == 0 ? 0 : PL + (az - 1) * RIM;
      St[(int64_t)(before + in_layer) * ld] = fac[j];
    }
    if (i == k && ucol) v = fmaf(alpha, tb.Mass[((size_t)e * Np + a) * Np + col], v);
    Su[(int64_t)a * ld] = v;
  }
}

// threads of a half: the columns of a pair, rounded up to warps
template <int NP1>
constexpr int hex32_half() {
  return (2 * NP1 * NP1 * NP1 - (NP1 - 2) * (NP1 - 2) * (NP1 - 2) + 31) / 32 * 32;
}

template <int NP1>
__global__ void __launch_bounds__(2 * hex32_half<NP1>(), NP1 == 5 ? 1 : (NP1 == 4 ? 2 : 5))
k_assemble_hex32(Dims dm, float alpha, RefTables ref, AsmTab<float> tb, float* __restrict__ S,
                 const double* __restrict__ rhs64, const __grid_constant__ Tab1D<NP1> tab) {
  constexpr int NQ1 = NP1 + 1, Np = NP1 * NP1 * NP1, Nb = Np - (NP1 - 2) * (NP1 - 2) * (NP1 - 2);
  constexpr int Nq = NQ1 * NQ1 * NQ1, Nfp = 6 * NQ1 * NQ1, H = hex32_half<NP1>(), Z = (NP1 + 1) / 2;
  __shared__ HexCoef<NP1> cs;
  const int tid = threadIdx.x, half = tid / H, c = tid % H;
  const int64_t e = blockIdx.x / 25, ld = dm.ld;
  const int pair = (int)(blockIdx.x % 25), i = pair / 5, k = pair % 5;
  const bool cq = !(i == 0 || (i <= 3 && k == 4)), ucol = c < Np;
  const size_t ep = (size_t)e * 25 + pair;
  const float *jv = tb.Jv + ep * (12 * Nq), *jf = tb.Jf + ep * (4 * Nfp);
  for (int q = tid; q < 12 * Nq; q += 2 * H) reinterpret_cast<float*>(cs.v)[(q % Nq) * 12 + q / Nq] = jv[q];
  for (int q = tid; q < 4 * Nfp; q += 2 * H) reinterpret_cast<float*>(cs.f)[(q % Nfp) * 4 + (q / Nfp + 3) % 4] = jf[q];
  for (int q = tid; q < Nfp; q += 2 * H)
    cs.fu[q] = tb.Su ? tb.Su[ep * Nfp + q] : (i == k ? tb.lamw[(size_t)e * Nfp + q] : 0.f);
  float* Se = S + e * (int64_t)dm.n * ld;
  if (pair == 0 && rhs64 != nullptr)
    for (int r = tid; r < dm.n; r += 2 * H) Se[r * ld + dm.n] = (float)rhs64[e * dm.n + r];
  __syncthreads();
  if (c >= Np + Nb) return;
  const int col = ucol ? c : c - Np;
  float* Sc = Se + (ucol ? k * Np + col : dm.nu + k * Nb + col);                 // this column
  float* Su = Sc + (int64_t)i * Np * ld;                                         // its u-rows
  float* St = Sc + (int64_t)(dm.nu + i * Nb) * ld;                               // its trace rows
  if (half == 0) hex32_layers<NP1, 0, Z>(cs, i, k, col, ucol, cq, e, ld, alpha, ref, tb, Su, St, tab);
  else hex32_layers<NP1, Z, NP1 - Z>(cs, i, k, col, ucol, cq, e, ld, alpha, ref, tb, Su, St, tab);
}

template <int NP1>
cudaError_t hex32_t(iedg_mesh* M, cudaStream_t st) {
  const Dims& dm = M->dm;
  Tab1D<NP1> tab;
  for (int g = 0; g <= NP1; ++g)
    for (int a = 0; a < NP1; ++a) {
      tab.L[g][a] = (float)M->L1h[(size_t)g * NP1 + a];
      tab.D[g][a] = (float)M->dL1h[(size_t)g * NP1 + a];
    }
  k_assemble_hex32<NP1><<<(unsigned)(M->E * 25), 2 * hex32_half<NP1>(), 0, st>>>(dm, (float)M->ph.alpha, M->ref,
                                                                                 tables32(M), M->S32, M->rhs64, tab);
  return cudaGetLastError();
}

template <class T, int D, int NP1>
cudaError_t col_t(iedg_mesh* M, T* S, const double* rhs64, const AsmTab<T>& tb, cudaStream_t st) {
  const int64_t n = M->E * M->dm.m * M->dm.m * (int64_t)(M->dm.Np + M->dm.Nb);
  k_assemble_col<T, D, NP1, NP1 + 1><<<(unsigned)((n + AC_THREADS - 1) / AC_THREADS), AC_THREADS, 0, st>>>(
      M->dm, M->ph, M->ref, tb, S, rhs64, M->E);
  return cudaGetLastError();
}

template <class T>
cudaError_t col_p(iedg_mesh* M, T* S, const double* rhs64, const AsmTab<T>& tb, cudaStream_t st) {
  if (M->dm.d == 3) return col_t<T, 3, 2>(M, S, rhs64, tb, st);
  if (M->dm.p == 1) return col_t<T, 2, 2>(M, S, rhs64, tb, st);
  if (M->dm.p == 2) return col_t<T, 2, 3>(M, S, rhs64, tb, st);
  return col_t<T, 2, 4>(M, S, rhs64, tb, st);
}

}  // namespace

bool assemble_col_supported(const iedg_mesh* M) {
  const Dims& dm = M->dm;
  if (M->tt.nb != nullptr || dm.nq1 != dm.p + 2) return false;
  if (dm.d == 2) return dm.p <= 3;
  return dm.p == 1 || (M->precision != 0 && dm.p <= 4);
}

cudaError_t launch_assemble_col(iedg_mesh* M, cudaStream_t st) {
  if (M->precision == 0) return col_p<double>(M, M->S, nullptr, tables64(M), st);
  if (M->dm.d == 3 && M->dm.p == 2) return hex32_t<3>(M, st);
  if (M->dm.d == 3 && M->dm.p == 3) return hex32_t<4>(M, st);
  if (M->dm.d == 3 && M->dm.p == 4) return hex32_t<5>(M, st);
  return col_p<float>(M, M->S32, M->rhs64, tables32(M), st);
}

}  // namespace iedg
