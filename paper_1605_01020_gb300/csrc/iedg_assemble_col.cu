// Element block assembly of small elements (2D of degree 1..3, 3D of degree 1, p + 2
// points per direction, uniform meshes): one thread per column of an (i, k) block.
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
  return M->tt.nb == nullptr && dm.nq1 == dm.p + 2 && (dm.d == 2 ? dm.p <= 3 : dm.p == 1);
}

cudaError_t launch_assemble_col(iedg_mesh* M, cudaStream_t st) {
  if (M->precision == 0) return col_p<double>(M, M->S, nullptr, tables64(M), st);
  return col_p<float>(M, M->S32, M->rhs64, tables32(M), st);
}

}  // namespace iedg
