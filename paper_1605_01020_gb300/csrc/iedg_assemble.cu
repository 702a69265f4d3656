// Element block assembly with the q-elimination folded in at the quadrature points,
// and the partial LU of the bordered element matrix (static condensation, Eq. LS).
//
// Bordered element matrix (rows x cols = n x (n+1), n = m Np + m Nb):
//     [ At  Bt  Ft ]     rows i Np + a      (u-equation i, node a)
//     [ Ct  Dt  Gt ]     rows nu + i Nb + s (trace equation i, slot s)
// columns k Np + b (u unknown k, node b), nu + k Nb + t (trace unknown k, slot t), n.
// A_qq = M (x) I (Eq. IEDG a) lets q be eliminated exactly:
//   dq_kl = M^-1 F_q,kl - G_l du_k + H_l dU_k,
// so with the lifted operators Gl(g) = Phi G_l, Hl(g) = Phi H_l at the points,
//   At_ik[a][b] = alpha delta_ik M_ab
//              + sum_{g,r} Dxi_r[g][a] (cu_ikr(g) Phi[g][b] - sum_l cq_iklr(g) Gl_l(g)[b])
//              + sum_fp PhiF[fp][a] (lamw delta_ik PhiF[fp][b] - sum_l fq_ikl(fp) GlF_l(fp)[b])
//   Bt_ik[a][t] = sum_{g,r} Dxi_r[g][a] sum_l cq_iklr(g) Hl_l(g)[t]
//              + sum_fp PhiF[fp][a] (fuh_ik(fp) mu_t(fp) + sum_l fq_ikl(fp) HlF_l(fp)[t])
// and the trace rows Ct, Dt equal the face parts of the u-rows of the boundary nodes
// (mu_s = phi_bnode[s] on every face), which is how they are formed here.
// The right-hand-side column is written by the point kernel: Ft = -R_u(u, q*),
// Gt = -R_FL,e(u, q*) (exact because the fluxes are affine in q).
#include "iedg_digits.cuh"
#include "iedg_internal.cuh"
#include "iedg_lu_common.cuh"
#include "iedg_tc.cuh"

namespace iedg {
namespace {

constexpr int AS_THREADS = 256;
constexpr int TM = 4, TN = 8;       // register tile of the volume contraction
constexpr int GC = 8;               // volume points per K-chunk

struct AsmCfg {
  int rows_pad;   // Np rounded up to TM
  int rg;         // row groups
  int CW;         // columns per CTA (multiple of TN)
  int cg;         // column groups
  int nsplit;     // CTAs per (element, i, k)
  int KC;         // K-chunk rows = GC d
};

AsmCfg asm_cfg(const Dims& dm) {
  AsmCfg c;
  c.rows_pad = idiv_up(dm.Np, TM) * TM;
  c.rg = c.rows_pad / TM;
  int max_cg = AS_THREADS / c.rg;
  int need = idiv_up(dm.Np + dm.Nb, TN);
  c.nsplit = idiv_up(need, max_cg);
  c.cg = idiv_up(need, c.nsplit);
  c.CW = c.cg * TN;
  c.KC = GC * dm.d;
  return c;
}

// T = double: FP64 path.  T = float: mixed path (FP32 element matrix; the FP64
// right-hand sides are copied into column n by one CTA per element).
// Meshes with mixed orders (tt.nb set): per-element slot count, offset and leading
// dimension; the trace basis at the face points comes from the element's table, and
// the trace rows are accumulated separately from the face parts of the u-rows.
template <class T, bool LIST = false>
__global__ void __launch_bounds__(AS_THREADS)
k_assemble(Dims dm, Phys ph, AsmCfg cf, RefTables ref, AsmTab<T> tb, T* __restrict__ S,
           const double* __restrict__ rhs64, TraceTab tt, int NbU, const int64_t* __restrict__ elist) {
  extern __shared__ __align__(16) unsigned char smraw[];
  T* sm = reinterpret_cast<T*>(smraw);
  const int tid = threadIdx.x;
  const int m2 = dm.m * dm.m;
  // the m^2 CTAs of an element are adjacent; with an element list (FP64 fallback of the
  // mixed path) CTA group `slot` assembles element elist[slot] into matrix slot `slot`
  const int64_t slot = blockIdx.x / m2;
  int64_t e = slot;
  if constexpr (LIST) {
    e = elist[slot];
    if (e < 0) return;
  }
  const int pair = blockIdx.x % m2, i = pair / dm.m, k = pair % dm.m;
  const int c0 = blockIdx.y * cf.CW;
  const int d = dm.d, Np = dm.Np, Nq = dm.Nq, Nfp = dm.Nfp, Nfq = dm.Nfq, Nfn = dm.Nfn;
  const bool mix = tt.nb != nullptr;
  const int NbT = dm.Nb;                            // slot stride of the lifting tables
  const int Nb = mix ? tt.nb[e] : dm.Nb;            // trace slots of this element
  const int ncol = Np + Nb;
  const int KC = cf.KC, CW = cf.CW, RP = cf.rows_pad;
  T* sA = sm;                           // [KC][RP]   Dxi_r[g][a]
  T* sB = sA + KC * RP;                 // [KC][CW]   W[(g, r)][col]
  T* facc = sB + KC * CW;               // [NbU][CW]  face parts of the boundary rows
  T* sV = facc + NbU * CW;              // [Nfq][CW]  face right operand
  T* tacc = mix ? sV + Nfq * CW : facc; // [Nb][CW]   trace rows (mixed orders), else = facc
  const T* mutab = nullptr;
  if (mix) {
    if constexpr (sizeof(T) == 8) mutab = reinterpret_cast<const T*>(tt.muf);
    else mutab = reinterpret_cast<const T*>(tt.muf32);
    mutab += (size_t)e * dm.nf * Nfq * tt.NFS;
  }
  const size_t jvs = (size_t)(1 + d) * d * Nq;
  const T* jv = tb.Jv + ((size_t)e * dm.m * dm.m + pair) * jvs;
  const size_t jfs = (size_t)(1 + d) * Nfp;
  const T* jf = tb.Jf + ((size_t)e * dm.m * dm.m + pair) * jfs;
  const T* GlV = tb.GlV + (size_t)e * d * Nq * Np;
  const T* HlV = tb.HlV + (size_t)e * d * Nq * NbT;
  const T* GlF = tb.GlF + (size_t)e * d * Nfp * Np;
  const T* HlF = tb.HlF + (size_t)e * d * Nfp * NbT;

  const int trow = tid / cf.cg, tcol = tid % cf.cg;
  const bool gemm_thread = trow < cf.rg;
  T acc[TM][TN];
#pragma unroll
  for (int a = 0; a < TM; ++a)
#pragma unroll
    for (int b = 0; b < TN; ++b) acc[a][b] = (T)0;

  // ---- volume contraction, K = Nq d in chunks of GC points
  for (int g0 = 0; g0 < Nq; g0 += GC) {
    for (int idx = tid; idx < KC * RP; idx += AS_THREADS) {
      int kc = idx / RP, a = idx % RP;
      int g = g0 + kc / d, r = kc % d;
      sA[idx] = (g < Nq && a < Np) ? tb.Dxi[((size_t)r * Nq + g) * Np + a] : (T)0;
    }
    for (int idx = tid; idx < KC * CW; idx += AS_THREADS) {
      int kc = idx / CW, col = c0 + idx % CW;
      int g = g0 + kc / d, r = kc % d;
      T w = 0;
      if (g < Nq && col < ncol) {
        if (col < Np) {
          w = jv[(size_t)r * Nq + g] * tb.Phi[(size_t)g * Np + col];
          for (int l = 0; l < d; ++l)
            w -= jv[(size_t)(d + l * d + r) * Nq + g] * GlV[((size_t)l * Nq + g) * Np + col];
        } else {
          for (int l = 0; l < d; ++l)
            w += jv[(size_t)(d + l * d + r) * Nq + g] * HlV[((size_t)l * Nq + g) * NbT + (col - Np)];
        }
      }
      sB[idx] = w;
    }
    __syncthreads();
    if (gemm_thread) {
      for (int kc = 0; kc < KC; ++kc) {
        T av[TM], bv[TN];
#pragma unroll
        for (int a = 0; a < TM; ++a) av[a] = sA[kc * RP + trow * TM + a];
#pragma unroll
        for (int b = 0; b < TN; ++b) bv[b] = sB[kc * CW + tcol * TN + b];
#pragma unroll
        for (int a = 0; a < TM; ++a)
#pragma unroll
          for (int b = 0; b < TN; ++b) acc[a][b] = fma(av[a], bv[b], acc[a][b]);
      }
    }
    __syncthreads();
  }

  // ---- face parts, accumulated per trace slot
  for (int idx = tid; idx < NbU * CW; idx += AS_THREADS) facc[idx] = (T)0;
  if (mix)
    for (int idx = tid; idx < Nb * CW; idx += AS_THREADS) tacc[idx] = (T)0;
  const T lamsel = (i == k) ? (T)1 : (T)0;
  for (int f = 0; f < dm.nf; ++f) {
    __syncthreads();
    for (int idx = tid; idx < Nfq * CW; idx += AS_THREADS) {
      int gf = idx / CW, col = c0 + idx % CW;
      int fp = f * Nfq + gf;
      T v = 0;
      if (col < Np) {
        // dfhat/du: lambda I (Lax-Friedrichs) or the pair's entry of S (Roe-type)
        const T su = tb.Su ? tb.Su[((size_t)e * dm.m * dm.m + pair) * Nfp + fp] : lamsel * tb.lamw[e * Nfp + fp];
        v = su * tb.PhiF[(size_t)fp * Np + col];
        for (int l = 0; l < d; ++l) v -= jf[(size_t)(1 + l) * Nfp + fp] * GlF[((size_t)l * Nfp + fp) * Np + col];
      } else if (col < ncol) {
        int t = col - Np;
        T mu = 0;
        if (mix) {
          const int* fl = tt.sfl + ((size_t)e * NbT + t) * 3;
          for (int q = 0; q < 3; ++q) {
            const int code = fl[q];
            if (code >= 0 && code / tt.NFS == f) mu = mutab[((size_t)f * Nfq + gf) * tt.NFS + code % tt.NFS];
          }
        } else {
          mu = tb.PhiF[(size_t)fp * Np + ref.bnode[t]];
        }
        v = jf[fp] * mu;
        for (int l = 0; l < d; ++l) v += jf[(size_t)(1 + l) * Nfp + fp] * HlF[((size_t)l * Nfp + fp) * NbT + t];
      }
      sV[idx] = v;
    }
    __syncthreads();
    for (int idx = tid; idx < Nfn * CW; idx += AS_THREADS) {
      int tn = idx / CW, cc = idx % CW;
      int a = ref.fnode[f * Nfn + tn];
      T s = 0;
      for (int gf = 0; gf < Nfq; ++gf) s += tb.PhiF[(size_t)(f * Nfq + gf) * Np + a] * sV[gf * CW + cc];
      facc[ref.slot[a] * CW + cc] += s;
    }
    if (mix) {
      // domain-boundary face: the trace rows take the boundary flux, so the right
      // operand is rebuilt from its derivatives
      if (tt.fkind && tt.fkind[e * dm.nf + f] != kFaceInterior) {
        __syncthreads();
        const int nc = 2 + d;
        for (int idx = tid; idx < Nfq * CW; idx += AS_THREADS) {
          int gf = idx / CW, col = c0 + idx % CW;
          int fp = f * Nfq + gf;
          const T* jb = tb.Jb + ((size_t)e * dm.m * dm.m + pair) * nc * Nfp + fp;
          T v = 0;
          if (col < Np) {
            v = jb[(size_t)Nfp] * tb.PhiF[(size_t)fp * Np + col];
            for (int l = 0; l < d; ++l) v -= jb[(size_t)(2 + l) * Nfp] * GlF[((size_t)l * Nfp + fp) * Np + col];
          } else if (col < ncol) {
            int t = col - Np;
            T mu = 0;
            const int* fl = tt.sfl + ((size_t)e * NbT + t) * 3;
            for (int q = 0; q < 3; ++q) {
              const int code = fl[q];
              if (code >= 0 && code / tt.NFS == f) mu = mutab[((size_t)f * Nfq + gf) * tt.NFS + code % tt.NFS];
            }
            v = jb[0] * mu;
            for (int l = 0; l < d; ++l) v += jb[(size_t)(2 + l) * Nfp] * HlF[((size_t)l * Nfp + fp) * NbT + t];
          }
          sV[idx] = v;
        }
        __syncthreads();
      }
      // trace rows: the slots living on this face, with the element's trace basis
      const int cnt = tt.nfs[e * dm.nf + f];
      const int* fsf = tt.fs + ((size_t)e * dm.nf + f) * tt.NFS;
      for (int idx = tid; idx < cnt * CW; idx += AS_THREADS) {
        int j = idx / CW, cc = idx % CW;
        T s = 0;
        for (int gf = 0; gf < Nfq; ++gf) s += mutab[((size_t)f * Nfq + gf) * tt.NFS + j] * sV[gf * CW + cc];
        tacc[fsf[j] * CW + cc] += s;
      }
    }
  }
  __syncthreads();

  // ---- write the element rows
  const int64_t nn = mix ? (int64_t)dm.nu + (int64_t)dm.m * Nb : dm.n;
  const int64_t ld = mix ? tt.ldv[e] : dm.ld;
  T* Se = mix ? S + tt.soff[e] : S + (LIST ? slot : e) * nn * ld;
  if (rhs64 != nullptr && pair == 0 && blockIdx.y == 0)
    for (int r = tid; r < nn; r += AS_THREADS) Se[r * ld + nn] = (T)rhs64[e * dm.n + r];
  auto colS = [&](int col) -> int64_t { return col < Np ? (int64_t)k * Np + col : (int64_t)dm.nu + (int64_t)k * Nb + (col - Np); };
  if (gemm_thread) {
    const T* Ms = tb.Mass + (size_t)e * Np * Np;
#pragma unroll
    for (int a = 0; a < TM; ++a) {
      int row = trow * TM + a;
      if (row >= Np) continue;
      int sl = ref.slot[row];
#pragma unroll
      for (int b = 0; b < TN; ++b) {
        int col = c0 + tcol * TN + b;
        if (col >= ncol || col >= c0 + CW) continue;
        T v = acc[a][b];
        if (sl >= 0) v += facc[sl * CW + (col - c0)];
        if (i == k && col < Np) v += (T)ph.alpha * Ms[row * Np + col];
        Se[((int64_t)i * Np + row) * ld + colS(col)] = v;
      }
    }
  }
  for (int idx = tid; idx < Nb * CW; idx += AS_THREADS) {
    int s = idx / CW, col = c0 + idx % CW;
    if (col >= ncol) continue;
    Se[((int64_t)dm.nu + (int64_t)i * Nb + s) * ld + colS(col)] = tacc[idx];
  }
}

// ------------------------------------------------------------------ partial LU
// Right-looking blocked LU with partial pivoting of the bordered matrix, pivots
// only among the nu u-rows (largest |a|, smallest row on ties), eliminating the
// first nu columns from all n rows.  Afterwards rows [nu, n) x cols [nu, n] hold
// [K_e | R_e] = [Dt - Ct At^-1 Bt | Gt - Ct At^-1 Ft]; rows [0, nu) hold U (upper
// triangle, cols < nu) and L^-1 P [Bt Ft] (cols >= nu) for the back-substitution.
// T = float (mixed path) additionally writes back every panel in full (the
// multipliers L, in the row order of their own panel step) and the pivot rows, for
// the refinement solves.
// A[r][c] -= sum_j L[r][j] U[j][c] over rows [r_lo, r_hi), cols [c_lo, c_hi): L from the
// row-major panel P (row r at P[(r - kb) NB + j]), U = rows kb..kb+nb of A, staged by
// UCW-column chunks in Uc; 16 x 16 threads with 4 x 4 register tiles.
template <class T, int NB>
__device__ __forceinline__ void lu64_update_rect(T* __restrict__ A, int ld, const T* __restrict__ P,
                                                 T* __restrict__ Uc, int kb, int nb, int r_lo, int r_hi, int c_lo,
                                                 int c_hi) {
  const int tid = threadIdx.x;
  for (int cc = c_lo; cc < c_hi; cc += UCW) {
    const int cw = min(UCW, c_hi - cc);
    for (int idx = tid; idx < NB * UCW; idx += LU_THREADS) {
      int j = idx / UCW, c = idx % UCW;
      Uc[idx] = (j < nb && c < cw) ? A[(int64_t)(kb + j) * ld + cc + c] : (T)0;
    }
    __syncthreads();
    const int tc = tid % (UCW / 4), tr = tid / (UCW / 4);   // 16 x 16 threads, 4x4 tiles
    for (int rb = r_lo; rb < r_hi; rb += 64) {
      T a4[4][4];
      int rr[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        rr[a] = rb + tr * 4 + a;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          int c = tc * 4 + b;
          a4[a][b] = (rr[a] < r_hi && c < cw) ? A[(int64_t)rr[a] * ld + cc + c] : (T)0;
        }
      }
      for (int j = 0; j < nb; ++j) {
        T uv[4], lv[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) uv[b] = Uc[j * UCW + tc * 4 + b];
#pragma unroll
        for (int a = 0; a < 4; ++a) lv[a] = rr[a] < r_hi ? P[(rr[a] - kb) * NB + j] : (T)0;
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) a4[a][b] = fma(-lv[a], uv[b], a4[a][b]);
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          int c = tc * 4 + b;
          if (rr[a] < r_hi && c < cw) A[(int64_t)rr[a] * ld + cc + c] = a4[a][b];
        }
    }
    __syncthreads();
  }
}

// |v| as a signed integer that orders like |v| (IEEE bit patterns of non-negative
// values are monotonic), -1 for NaN so that NaN is never chosen, like a floating-point
// comparison would; the pivot search of the FP64 LU then runs on the integer pipes
// instead of the slow FP64 pipe.
template <class T>
__device__ __forceinline__ long long abs_key(T v) {
  if constexpr (sizeof(T) == 8) {
    const long long k = __double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFLL;
    return k > 0x7FF0000000000000LL ? -1LL : k;
  } else {
    const long long k = (long long)(__float_as_int(v) & 0x7FFFFFFF);
    return k > 0x7F800000LL ? -1LL : k;
  }
}

// abs_key of +infinity: keys at or above it (and the -1 of NaN) are non-finite values
template <class T>
__device__ __forceinline__ long long inf_key() {
  if constexpr (sizeof(T) == 8) return 0x7FF0000000000000LL;
  else return 0x7F800000LL;
}

template <class T, int NB>
__device__ __forceinline__ void lu_element(const LuElem& el, T* __restrict__ S, int8_t* __restrict__ status,
                                           int* __restrict__ pivots, const int64_t e) {
  extern __shared__ __align__(16) unsigned char smraw[];
  T* sm = reinterpret_cast<T*>(smraw);
  __shared__ int piv[NB];
  __shared__ int perm[LU_MAX_NU];   // net row permutation of the current panel's interchanges
  __shared__ long long rv[LU_THREADS / 32];
  __shared__ int ri[LU_THREADS / 32];
  __shared__ int sing;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = el.n, nu = el.nu, ld = el.ld, ncol = n + 1;
  T* A = S + el.off;
  T* P = sm;                            // [n][NB]
  int nonfin = 0;                       // a pivot candidate was NaN or infinite
  T* Uc = P + (size_t)n * NB;           // [NB][UCW]
  if (tid == 0) sing = 0;
  for (int kb = 0; kb < nu; kb += NB) {
    const int nb = min(NB, nu - kb), rows = n - kb, prow = nu - kb;
    for (int idx = tid; idx < rows * NB; idx += LU_THREADS) {
      int r = idx / NB, j = idx % NB;
      P[idx] = j < nb ? A[(int64_t)(kb + r) * ld + kb + j] : (T)0;
    }
    for (int r = tid; r < prow; r += LU_THREADS) perm[r] = r;
    __syncthreads();
    for (int j = 0; j < nb; ++j) {
      long long best = -1;                  // largest |a| as an ordered integer key
      int bi = j;
      for (int r = j + tid; r < prow; r += LU_THREADS) {
        const long long v = abs_key(P[r * NB + j]);
        nonfin |= v < 0 || v >= inf_key<T>();
        if (v > best) { best = v; bi = r; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const long long ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
      }
      if (lane == 0) { rv[warp] = best; ri[warp] = bi; }
      __syncthreads();
      // every thread combines the warps' candidates (same order, same result)
      long long bk = rv[0];
      int pr = ri[0];
      for (int w = 1; w < LU_THREADS / 32; ++w) {
        const long long k = rv[w];
        if (k > bk || (k == bk && ri[w] < pr)) { bk = k; pr = ri[w]; }
      }
      if (bk <= 0) pr = j;                  // no nonzero candidate: singular
      if (tid == 0) {
        if (bk <= 0) sing = 1;
        piv[j] = pr;
        if (pivots) pivots[el.poff + kb + j] = kb + pr;
        if (pr != j) { const int t = perm[j]; perm[j] = perm[pr]; perm[pr] = t; }
      }
      if (pr != j && tid < NB) {
        T t = P[j * NB + tid];
        P[j * NB + tid] = P[pr * NB + tid];
        P[pr * NB + tid] = t;
      }
      __syncthreads();
      const T pv = P[j * NB + j];
      const T inv = pv != (T)0 ? (T)1 / pv : (T)0;
      for (int r = j + 1 + tid; r < rows; r += LU_THREADS) {
        T l = P[r * NB + j] * inv;
        P[r * NB + j] = l;
        for (int c = j + 1; c < nb; ++c) P[r * NB + c] = fma(-l, P[j * NB + c], P[r * NB + c]);
      }
      __syncthreads();
    }
    // U11 / L11 (and, when the factors are kept, L21) back to the element matrix
    const int wrows = pivots ? rows : nb;
    for (int idx = tid; idx < wrows * nb; idx += LU_THREADS) {
      int r = idx / nb, j = idx % nb;
      A[(int64_t)(kb + r) * ld + kb + j] = P[r * NB + j];
    }
    // trailing columns: row interchanges, then U12 = L11^-1 A12.  The panel's
    // interchanges leave row r holding the original row perm[r]; the rows below the
    // panel that change are pivot rows piv[j] >= nb and receive original rows above nb.
    // Each column gathers its new top rows (independent loads), moves the displaced
    // rows in groups of 8, then stores the top rows.
    for (int c = kb + nb + tid; c < ncol; c += LU_THREADS) {
      T x[NB];
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        if (j >= nb) break;
        x[j] = A[(int64_t)(kb + perm[j]) * ld + c];
      }
#pragma unroll
      for (int j0 = 0; j0 < NB; j0 += 8) {
        T y[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int r = j0 + j < nb ? piv[j0 + j] : 0;
          y[j] = (j0 + j < nb && r >= nb && perm[r] != r) ? A[(int64_t)(kb + perm[r]) * ld + c] : (T)0;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int r = j0 + j < nb ? piv[j0 + j] : 0;
          if (j0 + j < nb && r >= nb && perm[r] != r) A[(int64_t)(kb + r) * ld + c] = y[j];
        }
      }
      for (int j = 0; j < nb; ++j) {
        T s = x[j];
        for (int jj = 0; jj < j; ++jj) s = fma(-P[j * NB + jj], x[jj], s);
        x[j] = s;
        A[(int64_t)(kb + j) * ld + c] = s;
      }
    }
    __syncthreads();
    // A22 -= L21 U12, rows [kb+nb, n), cols [kb+nb, n]
    lu64_update_rect<T, NB>(A, ld, P, Uc, kb, nb, kb + nb, n, kb + nb, ncol);
  }
  // status: a non-finite pivot candidate, an exact zero pivot, or a non-finite Schur
  // complement
  nonfin = __syncthreads_or(nonfin);
  int bad = 0;
  for (int idx = tid; idx < (n - nu) * (ncol - nu); idx += LU_THREADS) {
    int r = nu + idx / (ncol - nu), c = nu + idx % (ncol - nu);
    if (!isfinite(A[(int64_t)r * ld + c])) bad = 1;
  }
  bad = __syncthreads_or(bad);
  if (tid == 0)
    status[e] = nonfin ? IEDG_ELEM_NONFINITE
                       : (sing ? IEDG_ELEM_SINGULAR : (bad ? IEDG_ELEM_NONFINITE : IEDG_ELEM_OK));
}

// ------------------------------------------------------------------ FP64 partial LU, digit form
// FP64 partial LU of the bordered element matrices with every trailing update on the
// tensor cores, by splitting the FP64 operands into 8-bit digits.
//
// Same factorisation as lu_element<double>: right-looking, 32-column
// panels, pivots among the u-rows only (largest |a|, lowest row on ties).  GB300 issues
// two FP64 multiply-adds per SM and clock against 4096 BF16 ones on the tensor cores,
// so the bulk of the arithmetic, A22 -= L21 U12 (rows x 32 times 32 x columns), goes
// there in integers:
//   * the panel's unknowns are scaled by powers of two, u_kj 2^-s_k and l_ik 2^s_k, so that
//     every row k of U12 has its largest entry near 1 (pivot rows of different equations
//     differ by powers of the Mach number); then each row of L21 and each column of U12 is
//     scaled by a power of two (by its largest entry) to integers |X| < 2^61 and cut into
//     eight balanced base-256 digits (iedg_digits.cuh), s = 0 the leading one, |d_0| <= 32;
//   * digit products of equal weight, s + t = l <= 8, share one FP32 accumulator in TMEM,
//     level 0 that of level 1 (256 d_0 is another slice of the row operand).  All sums are
//     integers below 2^24 (levels 0 and 1: 32 (32^2 256 + 2 32 128) < 2^23.1; the others
//     below 2^22), so the tensor core adds exactly (the splitting of Ozaki, Ogita, Oishi and
//     Rump, "Error-free transformations of matrix multiplication", 2012, with K short enough
//     that no level has to be flushed);
//   * the levels are joined in 96-bit integers, rounded once to FP64 and subtracted: one
//     FP64 addition per entry and panel where the DFMA form spends 32 multiply-adds.
// Accuracy.  The error of an update is absolute in its row and column: about 2^-60 times
// (largest |l_ik 2^s_k|) (largest |u_kj 2^-s_k|) over k, from rounding the operands and the
// levels past 8, at most 2^-54; then one FP64 rounding.  The DFMA form's is relative to the
// entry's own terms, 32 roundings of 2^-53.  So the digit form is the more accurate one for
// entries within about 2^-6 of that product, and the less accurate one far below it; entries
// whose old value and update are both below 2^-28 of it are formed by DFMA (0.4 % of them in
// the fourth line below, 1 % in the fifth, whose state has a direction at rest; 3 % of the
// kernel's time, 10 % with a line at 2^-20).
// Errors of K against 80-bit elimination, numpy model of both forms, DFMA | digits: largest
// entry, worst of the 25 component blocks, median entry:
//   p = 2, Re 2.5e5, M 0.2, cubes          2.2e-15 3.7e-13 4.6e-15 | 3.0e-16 2.7e-13 3.2e-15
//   p = 2, Re 1, M 0.02, cells 1 : 50      1.7e-15 1.5e-11 3.0e-14 | 2.1e-15 3.2e-12 2.0e-14
//   p = 2, Re 1, M 0.01, cells 1 : 1e4     7.5e-13 4.3e-07 1.7e-11 | 2.5e-13 3.9e-08 8.8e-12
//   p = 2, Re 1e-3, M 1e-4, cells 1 : 1000 1.3e-13 5.9e-07 1.0e-10 | 6.1e-14 3.4e-07 5.4e-11
//   p = 3, Re 2.5e5, M 0.2, cubes          3.6e-15 2.4e-13 2.2e-14 | 7.3e-16 1.7e-13 1.0e-14
//   p = 3, Re 10, M 0.05, cells 1 : 200    7.6e-15 1.9e-10 1.1e-13 | 5.6e-15 5.5e-11 5.3e-14
// (without s_k, level 8 and the rounding of the operands the second line's digits were
// 5.1e-15 1.8e-11 2.0e-13, the fourth's hundreds of times DFMA's).
//
// Roles: the 128 TMEM lanes are columns of A22 (the MMA's A operand is U12^T), so a
// warp's accesses of A22 are rows of 32 consecutive columns; the B operand stacks the
// digits t of 16 rows of L21, so that digit s of U12 meets all digits t <= 8 - s in one
// instruction whose columns land on the levels s .. 8 in order.
//
// Panel factorisation, the trace rows of L21 and U12 = L11^-1 A12 stay on the FP64 pipe,
// which bounds the kernel: per element of 320 + 280 unknowns 2.3 M multiply-adds there
// and 2 M additions of the updates (65 M multiply-adds in the DFMA form).  Two CTAs per
// SM, so that one element's panels overlap the other's updates.
// Measured, all elements of a mesh, DFMA form -> this one: 3D p = 3, 4096 elements
// 505.9 -> 102.1 ms; p = 2, 2002 elements 26.5 -> 7.9 ms; p = 4, 210 elements 238.6 -> 52.7 ms
// (without s_k, level 8, rounded operands and DFMA entries 96.0, 7.7, 48.4 ms);
// 2D p = 3 (64 + 48 unknowns), 851 elements 1.53 -> 0.84 ms.  Below 64 u-unknowns an
// element is at most two panels, which leaves too little to the tensor cores, and the
// DFMA form stays: 2D p = 2 (36 + 32), 1600 elements 0.79 ms DFMA, 0.98 ms digits; 3D p = 1
// (40 + 40), 8000 elements 4.98 and 5.10 ms.  Latency of the panel steps and of the
// trailing block's loads, not a pipe, is what is left.
constexpr int LT_NB = 32;                       // panel width
constexpr int LT_S = dig::S;                    // digits per operand, and levels kept
using dig::exponent_of;
constexpr int LT_ZERO = -4096;                  // exponent of a row or column of zeros
constexpr int LT_TC = 128, LT_TR = 16;          // columns and rows of one MMA group
constexpr int LT_RB = 64;                       // rows of L21 staged at a time
constexpr int LT_SLICE = LT_TC * LT_NB * 2;     // one digit of a column tile
constexpr int LT_A_BYTES = LT_S * LT_SLICE;     // 64 KB
constexpr int LT_BSLICE = LT_TR * LT_NB * 2;    // one digit of 16 rows
constexpr int LT_GROUP = (LT_S + 1) * LT_BSLICE;            // their digits 0..7, then 256 d_0
constexpr int LT_B_BYTES = LT_RB / LT_TR * LT_GROUP;        // 36 KB
constexpr int LT_LOW = 28;                      // entries below 2^-LT_LOW of row x column take DFMA
constexpr int LT_LVL_COLS = LT_S * LT_TR;       // TMEM columns of one accumulator set
constexpr int LT_TMEM_COLS = 2 * LT_LVL_COLS;   // two sets: epilogue of one, MMAs into the other
__host__ __device__ inline int lt_stride(int nu) { return nu | 1; }   // odd: conflict-free columns

__host__ inline size_t lt_smem(const Dims& dm) {
  const size_t panel = sizeof(double) * (size_t)LT_NB * lt_stride(dm.nu), dig = LT_A_BYTES + LT_B_BYTES;
  return (panel > dig ? panel : dig) + 128;      // operand tiles start on a 128-byte boundary
}

// sign s_k of eight of the panel's unknowns, from the largest exponents of their rows of U12.
__device__ __forceinline__ void load_shifts(const int* sk, int sign, int (&shift)[8]) {
  const int4 a = reinterpret_cast<const int4*>(sk)[0], b = reinterpret_cast<const int4*>(sk)[1];
  const int e[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
  for (int i = 0; i < 8; ++i) shift[i] = sign * (e[i] - 1023);
}

// Exponent with which a value that is scaled by 2^shift enters its row's or column's largest.
__device__ __forceinline__ int scaled_exp(double x, int shift) {
  const int e = exponent_of(x);
  return e == 0 ? LT_ZERO : (e == 0x7ff ? dig::BAD_EXP : e + shift);
}

// Digits of eight values scaled by 2^shift[i], emax the largest exponent then, |X| < 2^61:
// out(s, 8 packed BF16) for s = 0 (most significant) .. 7 and, TOP, 256 d_0 as s = 8.
template <bool TOP, class Out>
__device__ __forceinline__ void split8(const double (&x)[8], const int (&shift)[8], int emax, Out out) {
  uint32_t w[2][8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const unsigned long long v = dig::to_bytes(__double_as_longlong(x[i]), emax + 1 - shift[i]);
    w[0][i] = (uint32_t)(v >> 32);
    w[1][i] = (uint32_t)v;
  }
#pragma unroll
  for (int s = 0; s < LT_S; ++s) {
    const uint32_t(&q)[8] = w[s >> 2];
    out(s, make_uint4(dig::bf16_pair(q[0], q[1], s), dig::bf16_pair(q[2], q[3], s), dig::bf16_pair(q[4], q[5], s),
                      dig::bf16_pair(q[6], q[7], s)));
  }
  if constexpr (TOP) {
    const uint32_t(&q)[8] = w[0];
    out(LT_S, make_uint4(dig::bf16_pair(q[0], q[1], 0, 256.0f), dig::bf16_pair(q[2], q[3], 0, 256.0f),
                         dig::bf16_pair(q[4], q[5], 0, 256.0f), dig::bf16_pair(q[6], q[7], 0, 256.0f)));
  }
}

// One thread: all digit products of one 16-row group into the accumulator set at d (levels
// 0 and 1, then 2 .. 8); a, b: descriptors of the operands' first slices (addresses in their
// low bits, in 16 bytes).
__device__ __forceinline__ void lt_issue(uint32_t d, uint64_t a, uint64_t b, int ksteps) {
  auto mma = [&](int acc0, int s, int t, int nt, int ks, uint32_t add) {
    tc::mma_bf16(d + (uint32_t)(acc0 * LT_TR), a + (uint64_t)(s * (LT_SLICE >> 4) + ks * 16),
                 b + (uint64_t)(t * (LT_BSLICE >> 4) + ks * 16), tc::idesc_bf16(LT_TC, LT_TR * nt), add);
  };
  for (int ks = 0; ks < ksteps; ++ks) {
    mma(0, 1, 0, 8, ks, ks == 0 ? 0u : 1u);      // s = 1, t = 0..7: every accumulator
    mma(0, 0, 8, 1, ks, 1u);                     // s = 0, t = 0 by 256
    mma(0, 0, 1, 7, ks, 1u);                     // s = 0, t = 1..7
#pragma unroll
    for (int s = 2; s < LT_S; ++s) mma(s - 1, s, 0, 9 - s, ks, 1u);
  }
}

// minus the product sum whose accumulators are t[0..7] (256 level 0 + level 1, levels
// 2 .. 8), scales ef = row + column exponent.  Free of branches, so that a thread's eight
// entries overlap; `odd` is set where it cannot say: outside FP64's normal range, or below
// 2^32 units of the last level (2^-42 of row x column) and not zero.
__device__ __forceinline__ double join_levels(const float (&t)[8], int ef, bool& odd) {
  // integer-valued |t| <= 2^22 -> bits 0x4B400000 + t
  uint32_t b[8];
#pragma unroll
  for (int i = 1; i < 8; ++i) b[i] = __float_as_uint(t[i] + 12582912.0f);
  const int h = (int)((b[1] << 8) + b[2] - 0x8B400000u);        // 256 t1 + t2
  const int m = (int)((b[4] << 8) + b[5] - 0x8B400000u), n = (int)((b[6] << 8) + b[7] - 0x8B400000u);
  const long long L = (long long)m * 65536 + n;
  const long long H = (long long)__float2int_rn(t[0]) * (1 << 24) + (long long)h * 256 + (int)(b[3] - 0x4B400000u) + (L >> 32);
  // |H 2^32 + low word of L| (up to its last bit) in three words, normalised to two
  const uint32_t sg = (uint32_t)(int)(H >> 63);
  const uint32_t w2 = (uint32_t)((unsigned long long)H >> 32) ^ sg, w1 = (uint32_t)H ^ sg, w0 = (uint32_t)L ^ sg;
  const bool top = w2 != 0;
  const uint32_t x = top ? w2 : w1, y = top ? w1 : w0, z = top ? w0 : 0u;
  const int lz = __clz((int)x);
  const uint32_t hi = __funnelshift_l(y, x, lz), lo = __funnelshift_l(z, y, lz);
  const int field = ef - (top ? 1001 : 1033) - lz;              // biased exponent - 1
  const unsigned long long r = (((unsigned long long)hi << 21) | (lo >> 11)) + ((lo >> 10) & 1u) +
                               ((unsigned long long)(unsigned)field << 52);
  odd = x != 0 ? (unsigned)field >= 2045u : w0 != 0;
  return __longlong_as_double(x != 0 ? (long long)(r | ((unsigned long long)(~sg & 0x80000000u) << 32)) : 0ll);
}

// One entry of A22 by DFMA, in the DFMA form's order: l, u point to its row of L21 and its
// column of U12.
__device__ __forceinline__ double lt_entry(const double* l, const double* u, int ld, int nb, double a) {
#pragma unroll 4
  for (int k = 0; k < nb; ++k) a = fma(-l[k], u[(int64_t)k * ld], a);
  return a;
}

// Tensor-core state of a CTA, the same in every thread: bit b of phase is the parity of
// barrier b's next completion, bit b of pending says that a commit on it was not waited for.
struct LtTc {
  uint32_t tmem;
  uint64_t* mbar;
  uint32_t phase, pending;
  int failed, limit;
};

// Order of |v| as a signed integer, -1 for NaN (never chosen), as in the DFMA form.
__device__ __forceinline__ long long pivot_key(double v) {
  const long long k = __double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFLL;
  return k > 0x7FF0000000000000LL ? -1LL : k;
}

struct LtShared {
  int piv[LT_NB];
  double inv[LT_NB];                 // reciprocal pivots of the panel
  int perm[LU_MAX_NU];               // net row permutation of the panel's interchanges
  long long rv[LU_THREADS / 32];
  int ri[LU_THREADS / 32];
  int sing;
  alignas(16) int sk[LT_NB];         // largest exponents of the rows of U12: s_k = sk - 1023
  int ce[2][LT_TC];                  // column exponents, two halves of the panel's rows
  int re[LT_RB];                     // row exponents of the staged rows
  uint32_t cm[2][LT_TC], rm[LT_RB];  // which of the panel's 32 values are not zero
};

// Panel columns kb .. kb+nb-1 over the u-rows, P column-major (column j at P + j PR).
// Two barriers per column: the pass that applies column j's multipliers also finds
// column j+1's pivot candidates; one warp swaps the pivot rows, another forms the
// reciprocal once (an FP64 division in every thread would load the FP64 pipe).
__device__ __forceinline__ void lt_panel(LtShared& sh, double* P, int PR, int prow, int nb, int& nonfin) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr long long INF = 0x7FF0000000000000LL;
  for (int j = 0; j < nb; ++j) {
    long long best = -1;
    int bi = j;
    auto candidate = [&](double v, int r) {
      const long long k = pivot_key(v);
      nonfin |= k < 0 || k >= INF;
      if (k > best) { best = k; bi = r; }
    };
    if (j == 0) {
      for (int r = tid; r < prow; r += LU_THREADS) candidate(P[r], r);
    } else {
      const double inv = sh.inv[j - 1];
      const double* piv_row = P + (j - 1);
      for (int r = j + tid; r < prow; r += LU_THREADS) {
        double* row = P + r;
        const double l = row[(j - 1) * PR] * inv;
        row[(j - 1) * PR] = l;
        const double v = fma(-l, piv_row[j * PR], row[j * PR]);
        row[j * PR] = v;
        candidate(v, r);
        for (int c = j + 1; c < nb; ++c) row[c * PR] = fma(-l, piv_row[c * PR], row[c * PR]);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
    }
    if (lane == 0) { sh.rv[warp] = best; sh.ri[warp] = bi; }
    __syncthreads();
    if (warp < 2) {
      long long bk = sh.rv[0];
      int pr = sh.ri[0];
      for (int w = 1; w < LU_THREADS / 32; ++w) {
        const long long k = sh.rv[w];
        if (k > bk || (k == bk && sh.ri[w] < pr)) { bk = k; pr = sh.ri[w]; }
      }
      if (bk <= 0) pr = j;                  // no nonzero candidate: singular
      const double pv = P[pr + j * PR];
      if (warp == 1) {
        if (lane == 0) sh.inv[j] = pv != 0.0 ? 1.0 / pv : 0.0;
      }
      asm volatile("bar.sync 1, 64;" ::: "memory");   // pv read before the rows trade places
      if (warp == 0) {
        if (lane == 0) {
          if (bk <= 0) sh.sing = 1;
          sh.piv[j] = pr;
          if (pr != j) { const int t = sh.perm[j]; sh.perm[j] = sh.perm[pr]; sh.perm[pr] = t; }
        }
        if (pr != j) {
          const double t = P[j + lane * PR];
          P[j + lane * PR] = P[pr + lane * PR];
          P[pr + lane * PR] = t;
        }
      }
    }
    __syncthreads();
  }
  // the last column's multipliers
  const double inv = sh.inv[nb - 1];
  for (int r = nb + tid; r < prow; r += LU_THREADS) P[r + (nb - 1) * PR] *= inv;
  __syncthreads();
}

// A22 -= L21 U12 over rows [r0, n), columns [c0, ncol).  Returns false when a completion
// wait ran out.  `bad` collects non-finite results of the trace block (last panel).
__device__ __forceinline__ bool lt_trailing(LtShared& sh, double* __restrict__ A, int ld, int kb, int nb, int r0, int n,
                                            int nu, int c0, int ncol, unsigned char* dig, LtTc* tcs, int& bad) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int q = warp & 3, h = warp >> 2;
  unsigned char *da = dig, *db = dig + LT_A_BYTES;
  const uint64_t ua = tc::desc_kmajor(tc::smem_u32(da), 128, 512), ub = tc::desc_kmajor(tc::smem_u32(db), 128, 512);
  const int ksteps = nb > 16 ? 2 : 1;
  // L21 rows are staged by lane = row and eight of the panel's columns; the next 64 rows
  // are requested while the current ones are worked on
  const int srow = 8 * warp + (lane & 7), sk8 = lane >> 3;
  double x[8];
  auto fetch = [&](int row) {
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      const int k = 8 * sk8 + i;
      double2 t = make_double2(0.0, 0.0);
      if (row < n && k + 1 < nb) t = *reinterpret_cast<const double2*>(A + (int64_t)row * ld + kb + k);
      else if (row < n && k < nb) t.x = A[(int64_t)row * ld + kb + k];
      x[i] = t.x;
      x[i + 1] = t.y;
    }
  };
  fetch(r0 + srow);
  for (int ct = c0; ct < ncol; ct += LT_TC) {
    {
      // U12 columns ct .. ct+127: thread = column (and half of the panel's rows)
      const int c = tid & (LT_TC - 1), kh = tid >> 7, col = ct + c;
      double x[2][8];
      int em = LT_ZERO, shift[2][8];
      uint32_t nz = 0;
#pragma unroll
      for (int u = 0; u < 2; ++u) load_shifts(sh.sk + 16 * kh + 8 * u, -1, shift[u]);
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int k = 16 * kh + 8 * u + i;
          x[u][i] = (k < nb && col < ncol) ? A[(int64_t)(kb + k) * ld + col] : 0.0;
          const int e = scaled_exp(x[u][i], shift[u][i]);
          em = max(em, e);
          nz |= e != LT_ZERO ? 1u << (8 * u + i) : 0u;
        }
      sh.ce[kh][c] = em;
      sh.cm[kh][c] = nz << (16 * kh);
      __syncthreads();
      em = max(em, sh.ce[kh ^ 1][c]);
#pragma unroll
      for (int u = 0; u < 2; ++u)
        split8<false>(x[u], shift[u], em, [&](int s, uint4 v) {
          *reinterpret_cast<uint4*>(da + s * LT_SLICE + tc::core_off16(c, 16 * kh + 8 * u)) = v;
        });
    }
    const int c = 32 * q + lane, col = ct + c;
    int ecol = 0;                                    // set after the first barrier below
    uint32_t cmask = 0;
    for (int rb = r0; rb < n; rb += LT_RB) {
      {
        int em = LT_ZERO, shift[8];
        uint32_t nz = 0;
        load_shifts(sh.sk + 8 * sk8, 1, shift);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int e = scaled_exp(x[i], shift[i]);
          em = max(em, e);
          nz |= e != LT_ZERO ? 1u << (8 * sk8 + i) : 0u;
        }
        em = max(em, __shfl_xor_sync(0xffffffffu, em, 8));
        em = max(em, __shfl_xor_sync(0xffffffffu, em, 16));
        nz |= __shfl_xor_sync(0xffffffffu, nz, 8);
        nz |= __shfl_xor_sync(0xffffffffu, nz, 16);
        if (sk8 == 0) { sh.re[srow] = em; sh.rm[srow] = nz; }
        split8<true>(x, shift, em, [&](int s, uint4 v) {
          *reinterpret_cast<uint4*>(db + (srow >> 4) * LT_GROUP + s * LT_BSLICE +
                                    tc::core_off16(srow & 15, 8 * sk8)) = v;
        });
        fetch((rb + LT_RB < n ? rb + LT_RB : r0) + srow);
      }
      tc::fence_proxy_async();
      __syncthreads();
      tc::fence_after_sync();
      if (rb == r0) {
        ecol = max(sh.ce[0][c], sh.ce[1][c]);
        cmask = sh.cm[0][c] | sh.cm[1][c];
      }
      const int ng = (min(LT_RB, n - rb) + LT_TR - 1) / LT_TR;
      if (tid == 0) {
        lt_issue(tcs->tmem, ua, ub, ksteps);
        tc::mma_commit(tcs->mbar);
      }
      tcs->pending |= 1u;
      for (int g = 0; g < ng; ++g) {
        const int b = g & 1;
        if (g + 1 < ng) {        // the other accumulator set was read before the last barrier
          if (tid == 0) {
            lt_issue(tcs->tmem + (uint32_t)((b ^ 1) * LT_LVL_COLS), ua, ub + (uint64_t)((g + 1) * (LT_GROUP >> 4)), ksteps);
            tc::mma_commit(tcs->mbar + (b ^ 1));
          }
          tcs->pending |= 1u << (b ^ 1);
        }
        // this thread's column, rows 8h .. 8h+7 of the group
        const int row0 = rb + LT_TR * g + 8 * h;
        double* dst = A + (int64_t)row0 * ld + col;
        double a[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) a[i] = (col < ncol && row0 + i < n) ? dst[(int64_t)i * ld] : 0.0;
        const bool ok = tc::mbar_wait(tcs->mbar + b, (tcs->phase >> b) & 1u, tcs->limit);
        if (ok) {
          tc::fence_after_sync();
          float t[8][8];
          dig::load_levels(tcs->tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * LT_LVL_COLS + 8 * h), LT_TR, t);
          // entries for DFMA: those join_levels cannot say, with non-finite operands, or far below
          // row x column
          unsigned redo = 0;
          double d[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float lv[8] = {t[0][i], t[1][i], t[2][i], t[3][i], t[4][i], t[5][i], t[6][i], t[7][i]};
            const int lr = LT_TR * g + 8 * h + i, ef = ecol + sh.re[lr];
            bool odd;
            d[i] = join_levels(lv, ef, odd);
            const int eo = max(exponent_of(a[i]), exponent_of(d[i]));
            if (odd || eo <= ef - 1022 - LT_LOW) redo |= 1u << i;
            d[i] += a[i];
          }
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (col < ncol && row0 + i < n && !((redo >> i) & 1u)) {
              dst[(int64_t)i * ld] = d[i];
              bad |= row0 + i >= nu && col >= nu && exponent_of(d[i]) == 0x7ff;
            }
          for (; redo; redo &= redo - 1) {
            const int row = row0 + __ffs(redo) - 1, lr = row - rb;
            // products that all vanish leave the entry as it is, unless an operand is not finite
            if (col >= ncol || row >= n || ((cmask & sh.rm[lr]) == 0 && max(ecol, sh.re[lr]) < dig::BAD_EXP)) continue;
            double* v = A + (int64_t)row * ld + col;
            *v = lt_entry(A + (int64_t)row * ld + kb, A + (int64_t)kb * ld + col, ld, nb, *v);
            bad |= row >= nu && col >= nu && exponent_of(*v) == 0x7ff;
          }
        }
        tc::fence_before_sync();
        if (__syncthreads_or(!ok)) { tcs->failed = 1; return false; }
        tc::fence_after_sync();
        tcs->phase ^= 1u << b;
        tcs->pending &= ~(1u << b);
      }
    }
  }
  return true;
}

__device__ __forceinline__ bool lt_element(LtShared& sh, const LuElem& el, double* __restrict__ S,
                                           int8_t* __restrict__ status, int64_t e, unsigned char* smem, LtTc* tcs) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = el.n, nu = el.nu, ld = el.ld, ncol = n + 1;
  double* A = S + el.off;
  double* P = reinterpret_cast<double*>(smem);
  const int PR = lt_stride(nu);
  int nonfin = 0, bad = 0;
  if (tid == 0) sh.sing = 0;
  for (int kb = 0; kb < nu; kb += LT_NB) {
    const int nb = min(LT_NB, nu - kb), prow = nu - kb;
    for (int r = warp; r < prow; r += LU_THREADS / 32)
      P[r + lane * PR] = lane < nb ? A[(int64_t)(kb + r) * ld + kb + lane] : 0.0;
    for (int r = tid; r < prow; r += LU_THREADS) sh.perm[r] = r;
    if (tid < LT_NB) sh.sk[tid] = 0;
    __syncthreads();
    lt_panel(sh, P, PR, prow, nb, nonfin);
    // [L11 \ U11], L21 of the u-rows back
    for (int r = warp; r < prow; r += LU_THREADS / 32)
      if (lane < nb) A[(int64_t)(kb + r) * ld + kb + lane] = P[r + lane * PR];
    // L21 of the trace rows, x U11 = a: one thread per row, no pivots among them
    for (int r = nu + tid; r < n; r += LU_THREADS) {
      double* row = A + (int64_t)r * ld + kb;
      double x[LT_NB];
      // rows start on 32-byte boundaries (ld and kb are multiples of 4)
#pragma unroll
      for (int j = 0; j < LT_NB; j += 2) {
        double2 t = make_double2(0.0, 0.0);
        if (j + 1 < nb) t = *reinterpret_cast<const double2*>(row + j);
        else if (j < nb) t.x = row[j];
        x[j] = t.x;
        x[j + 1] = t.y;
      }
#pragma unroll
      for (int j = 0; j < LT_NB; ++j) {
        if (j >= nb) break;
        x[j] *= sh.inv[j];
#pragma unroll
        for (int c = j + 1; c < LT_NB; ++c) x[c] = fma(-x[j], P[j + c * PR], x[c]);
      }
#pragma unroll
      for (int j = 0; j < LT_NB; j += 2) {
        if (j + 1 < nb) *reinterpret_cast<double2*>(row + j) = make_double2(x[j], x[j + 1]);
        else if (j < nb) row[j] = x[j];
      }
    }
    // trailing columns: row interchanges (each column gathers its new top rows, then
    // moves the displaced rows), then U12 = L11^-1 A12 and the largest exponents of its rows
    for (int c0 = kb + nb + 32 * warp; c0 < ncol; c0 += LU_THREADS) {
      const int c = c0 + lane;
      const bool in = c < ncol;
      double x[LT_NB];
#pragma unroll
      for (int j = 0; j < LT_NB; ++j) x[j] = (in && j < nb) ? A[(int64_t)(kb + sh.perm[j]) * ld + c] : 0.0;
#pragma unroll
      for (int j0 = 0; j0 < LT_NB; j0 += 8) {
        double y[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int r = j0 + j < nb ? sh.piv[j0 + j] : 0;
          y[j] = (in && j0 + j < nb && r >= nb && sh.perm[r] != r) ? A[(int64_t)(kb + sh.perm[r]) * ld + c] : 0.0;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int r = j0 + j < nb ? sh.piv[j0 + j] : 0;
          if (in && j0 + j < nb && r >= nb && sh.perm[r] != r) A[(int64_t)(kb + r) * ld + c] = y[j];
        }
      }
#pragma unroll
      for (int j = 0; j < LT_NB; ++j) {
        if (j >= nb) break;
#pragma unroll
        for (int i = j + 1; i < LT_NB; ++i) x[i] = fma(-P[i + j * PR], x[j], x[i]);
        if (in) A[(int64_t)(kb + j) * ld + c] = x[j];
      }
      int top = 0;                           // lane j keeps row j's
#pragma unroll
      for (int j = 0; j < LT_NB; ++j) {
        const int e = __reduce_max_sync(0xffffffffu, exponent_of(x[j]));
        top = lane == j ? e : top;
      }
      if (lane < nb) atomicMax(&sh.sk[lane], top);
    }
    __syncthreads();
    if (!lt_trailing(sh, A, ld, kb, nb, kb + nb, n, nu, kb + nb, ncol, smem, tcs, bad)) break;
    if (kb + nb < nu) bad = 0;                 // only the last panel's trace block is the Schur complement
    __syncthreads();
  }
  nonfin = __syncthreads_or(nonfin);
  bad = __syncthreads_or(bad);
  if (tid == 0)
    status[e] = tcs->failed ? IEDG_ELEM_TIMEOUT
                            : (nonfin ? IEDG_ELEM_NONFINITE
                                      : (sh.sing ? IEDG_ELEM_SINGULAR : (bad ? IEDG_ELEM_NONFINITE : IEDG_ELEM_OK)));
  return !tcs->failed;
}

// TMEM and the completion barriers are set up once per CTA; a CTA whose wait ran out
// factors nothing more, flags the elements it still takes from the queue, waits once
// more (bounded) for its MMAs in flight and frees its TMEM.
__global__ void __launch_bounds__(LU_THREADS, 2)
k_lu64_tc(Dims dm, LuDesc lud, double* __restrict__ S, int8_t* __restrict__ status, int64_t* queue, int64_t E,
          int* err, int wait_limit) {
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned char* smem = smraw + ((128u - (tc::smem_u32(smraw) & 127u)) & 127u);
  __shared__ LtShared sh;
  __shared__ uint32_t tmem_base;
  __shared__ __align__(8) uint64_t mbar[2];
  const int tid = threadIdx.x, warp = tid >> 5;
  if (warp == 0) {
    tc::tmem_alloc(&tmem_base, LT_TMEM_COLS);
    tc::tmem_relinquish();
  }
  if (tid == 0) {
    tc::mbar_init(&mbar[0], 1);
    tc::mbar_init(&mbar[1], 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  LtTc mine;
  mine.tmem = tmem_base;
  mine.mbar = mbar;
  mine.phase = mine.pending = 0;
  mine.failed = 0;
  mine.limit = wait_limit;
  int64_t e, it = 0;
  for (; next_element(queue, E, it, lud.order, &e); ++it) {
    if (!lt_element(sh, lu_elem(dm, lud, e), S, status, e, smem, &mine)) {
      if (tid == 0) atomicOr(err, 1);
      for (int b = 0; b < 2; ++b)      // MMAs still in flight finish before the TMEM is freed
        if ((mine.pending >> b) & 1u) tc::mbar_wait(mbar + b, (mine.phase >> b) & 1u, kTcWaitLimit);
      ++it;
      break;
    }
  }
  if (mine.failed)
    for (; next_element(queue, E, it, lud.order, &e); ++it)
      if (tid == 0) status[e] = IEDG_ELEM_TIMEOUT;
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tmem_base, LT_TMEM_COLS);
}

template <class T, int NB>
__global__ void __launch_bounds__(LU_THREADS)
k_lu(Dims dm, LuDesc lud, T* __restrict__ S, int8_t* __restrict__ status, int* __restrict__ pivots, int64_t* queue,
     int64_t E, const int64_t* __restrict__ active = nullptr) {
  int64_t e;
  for (int64_t it = 0; next_element(queue, E, it, lud.order, &e); ++it)
    if (active == nullptr || active[e] >= 0) lu_element<T, NB>(lu_elem(dm, lud, e), S, status, pivots, e);
}

}  // namespace

size_t lu64_smem(const Dims& dm, int nb);

template <class T>
static cudaError_t assemble_t(iedg_mesh* M, T* S, const double* rhs64, const AsmTab<T>& tb, cudaStream_t st) {
  const Dims& dm = M->dm;
  AsmCfg cf = asm_cfg(dm);
  const bool mix = M->tt.nb != nullptr;
  int inner = 1;
  for (int r = 0; r < dm.d; ++r) inner *= dm.p - 1;
  const int nbu = dm.Np - inner;                  // boundary nodes of the element
  size_t smem = sizeof(T) * ((size_t)cf.KC * cf.rows_pad + (size_t)cf.KC * cf.CW + (size_t)nbu * cf.CW +
                             (size_t)dm.Nfq * cf.CW + (mix ? (size_t)dm.Nb * cf.CW : 0));
  cudaError_t err = cudaFuncSetAttribute(k_assemble<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  dim3 grid((unsigned)(M->E * dm.m * dm.m), cf.nsplit);
  k_assemble<T><<<grid, AS_THREADS, smem, st>>>(dm, M->ph, cf, M->ref, tb, S, rhs64, M->tt, nbu, nullptr);
  return cudaGetLastError();
}

AsmTab<double> tables64(const iedg_mesh* M) {
  const Geo& G = M->geo;
  const PointJac& P = M->pj;
  return AsmTab<double>{M->ref.Phi, M->ref.Dxi, M->ref.PhiF, P.Jv, P.Jf, P.lamw, P.Su, P.Jb,
                        G.GlV, G.HlV, G.GlF, G.HlF, G.Mass};
}

AsmTab<float> tables32(const iedg_mesh* M) {
  const Geo& G = M->geo;
  const PointJac& P = M->pj;
  return AsmTab<float>{M->ref.Phi32, M->ref.Dxi32, M->ref.PhiF32, P.Jv32, P.Jf32, P.lamw32, P.Su32, P.Jb32,
                       G.GlV32, G.HlV32, G.GlF32, G.HlF32, G.Mass32};
}

cudaError_t launch_assemble_list(iedg_mesh* M, double* S, const int64_t* elist, int64_t n_slots, cudaStream_t st) {
  const Dims& dm = M->dm;
  if (assemble_dg_supported(dm)) return launch_assemble_dg(M, S, elist, n_slots, st);
  AsmCfg cf = asm_cfg(dm);
  int inner = 1;
  for (int r = 0; r < dm.d; ++r) inner *= dm.p - 1;
  const int nbu = dm.Np - inner;
  size_t smem = sizeof(double) * ((size_t)cf.KC * cf.rows_pad + (size_t)cf.KC * cf.CW + (size_t)nbu * cf.CW +
                                  (size_t)dm.Nfq * cf.CW);
  cudaError_t err =
      cudaFuncSetAttribute(k_assemble<double, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  dim3 grid((unsigned)(n_slots * dm.m * dm.m), cf.nsplit);
  k_assemble<double, true><<<grid, AS_THREADS, smem, st>>>(dm, M->ph, cf, M->ref, tables64(M), S, M->rhs64, M->tt,
                                                           nbu, elist);
  return cudaGetLastError();
}

cudaError_t launch_lu64_list(iedg_mesh* M, double* S, int64_t n_slots, const int64_t* active, int8_t* status,
                             cudaStream_t st) {
  const Dims& dm = M->dm;
  size_t smem = lu64_smem(dm, 16);
  cudaError_t err = cudaFuncSetAttribute(k_lu<double, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  k_lu<double, 16><<<(unsigned)n_slots, LU_THREADS, smem, st>>>(dm, LuDesc{}, S, status, nullptr, nullptr, n_slots,
                                                                active);
  return cudaGetLastError();
}

cudaError_t launch_assemble(iedg_mesh* M, cudaStream_t st) {
  if (M->precision == 0) return assemble_t<double>(M, M->S, nullptr, tables64(M), st);
  return assemble_t<float>(M, M->S32, M->rhs64, tables32(M), st);
}

template <class T, int NB>
static cudaError_t lu_t(iedg_mesh* M, T* S, int* piv, cudaStream_t st) {
  const Dims& dm = M->dm;
  size_t smem = sizeof(T) * ((size_t)dm.n * NB + (size_t)NB * UCW);
  cudaError_t err = cudaFuncSetAttribute(k_lu<T, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  if (M->sched.lu_persistent) {
    unsigned grid = 0;
    err = persistent_grid(k_lu<T, NB>, smem, M->E, &grid);
    if (err == cudaSuccess) err = cudaMemsetAsync(M->queue, 0, sizeof(int64_t), st);
    if (err != cudaSuccess) return err;
    k_lu<T, NB><<<grid, LU_THREADS, smem, st>>>(dm, M->lud, S, M->status, piv, M->queue, M->E);
  } else {
    k_lu<T, NB><<<(unsigned)M->E, LU_THREADS, smem, st>>>(dm, M->lud, S, M->status, piv, nullptr, M->E);
  }
  return cudaGetLastError();
}

size_t lu64_smem(const Dims& dm, int nb) { return sizeof(double) * ((size_t)dm.n * nb + (size_t)nb * UCW); }

static cudaError_t launch_lu64_tc(iedg_mesh* M, cudaStream_t st) {
  const size_t smem = lt_smem(M->dm);
  cudaError_t err = cudaFuncSetAttribute(k_lu64_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  unsigned grid = (unsigned)M->E;
  int64_t* queue = nullptr;
  if (M->sched.lu_persistent) {
    // two resident CTAs at most: each holds half of the SM's TMEM
    err = persistent_grid(k_lu64_tc, smem, M->E, &grid, 2);
    if (err == cudaSuccess) err = cudaMemsetAsync(M->queue, 0, sizeof(int64_t), st);
    if (err != cudaSuccess) return err;
    queue = M->queue;
  }
  k_lu64_tc<<<grid, LU_THREADS, smem, st>>>(M->dm, M->lud, M->S, M->status, queue, M->E, M->dev_flag,
                                            tc_wait_limit(M));
  return cudaGetLastError();
}

cudaError_t launch_lu(iedg_mesh* M, cudaStream_t st) {
  if (M->dm.nu > LU_MAX_NU) return cudaErrorInvalidValue;   // orders above 4 are rejected at creation
  if (M->precision == 0 && M->sched.lu_tensor) return launch_lu64_tc(M, st);
  if (M->precision == 0) {
    if (M->sched.lu_panel == 32 && lu64_smem(M->dm, 32) <= 227 * 1024) return lu_t<double, 32>(M, M->S, nullptr, st);
    return lu_t<double, 16>(M, M->S, nullptr, st);
  }
  if (M->schur_in == kSchurFp32 && M->sched.lu_tensor == 2) return launch_lu32_mma(M, M->dm.n, st);
  return launch_lu32(M, st);
}

}  // namespace iedg
