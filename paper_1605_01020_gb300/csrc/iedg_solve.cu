// Trace solve K dU = R (Eq. LS) on the GPU: restarted GMRES with iterated classical
// Gram-Schmidt (two CGS passes per Arnoldi step) and left preconditioning
// M^-1 K dU = M^-1 R, as in the paper's parallel solver (Sec. 2.2.2).  On one GPU
// there is one subdomain; the preconditioner here is block Jacobi with the m x m
// diagonal blocks of K (the paper notes that zero overlap gives block Jacobi), or
// BILU(0) in multicolour order.  The whole iteration is one cooperative launch (k_gmres).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "iedg_internal.cuh"

using namespace iedg;

namespace {

constexpr int SV_THREADS = 256;

// Dinv[t] = inverse of the diagonal block K[t][t] (Gauss-Jordan, partial pivoting).
__global__ void k_diag_inv(int m, int64_t T, const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                           const double* __restrict__ K, double* __restrict__ Dinv, int* __restrict__ flag) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= T) return;
  int64_t lo = row_ptr[t], hi = row_ptr[t + 1], blk = -1;
  while (lo < hi) {
    int64_t mid = (lo + hi) / 2;
    if (col[mid] < t) lo = mid + 1; else hi = mid;
  }
  if (lo < row_ptr[t + 1] && col[lo] == t) blk = lo;
  double a[5][10];
  for (int i = 0; i < m; ++i)
    for (int j = 0; j < 2 * m; ++j) a[i][j] = j < m ? (blk >= 0 ? K[(blk * m + i) * m + j] : 0.0) : (j - m == i);
  bool ok = blk >= 0;
  for (int c = 0; c < m && ok; ++c) {
    int pr = c;
    for (int r = c + 1; r < m; ++r)
      if (fabs(a[r][c]) > fabs(a[pr][c])) pr = r;
    if (a[pr][c] == 0.0) { ok = false; break; }
    if (pr != c)
      for (int j = 0; j < 2 * m; ++j) { double x = a[c][j]; a[c][j] = a[pr][j]; a[pr][j] = x; }
    double inv = 1.0 / a[c][c];
    for (int j = 0; j < 2 * m; ++j) a[c][j] *= inv;
    for (int r = 0; r < m; ++r) {
      if (r == c) continue;
      double f = a[r][c];
      for (int j = 0; j < 2 * m; ++j) a[r][j] -= f * a[c][j];
    }
  }
  if (!ok) atomicOr(flag, 1);
  for (int i = 0; i < m; ++i)
    for (int j = 0; j < m; ++j) Dinv[(t * m + i) * m + j] = ok ? a[i][m + j] : (i == j);
}

// ---------------------------------------------------------------- BILU(0)
// Rows of one colour, one CTA per row: for each neighbour k eliminated before the row
// (in elimination order), L_ik = A_ik U_kk^-1, then A_ij -= L_ik U_kj for the row's
// later entries j present in row k (threads over j, binary search in row k); finally
// the inverse of the row's diagonal block.  Rows of one colour share no block.
constexpr int BI_THREADS = 128;
__device__ bool invert_block(int m, const double* __restrict__ a_in, double* __restrict__ out) {
  double a[5][10];
  for (int i = 0; i < m; ++i)
    for (int j = 0; j < 2 * m; ++j) a[i][j] = j < m ? a_in[i * m + j] : (j - m == i);
  for (int c = 0; c < m; ++c) {
    int pr = c;
    for (int r = c + 1; r < m; ++r)
      if (fabs(a[r][c]) > fabs(a[pr][c])) pr = r;
    if (a[pr][c] == 0.0) return false;
    if (pr != c)
      for (int j = 0; j < 2 * m; ++j) { double x = a[c][j]; a[c][j] = a[pr][j]; a[pr][j] = x; }
    double inv = 1.0 / a[c][c];
    for (int j = 0; j < 2 * m; ++j) a[c][j] *= inv;
    for (int r = 0; r < m; ++r) {
      if (r == c) continue;
      double f = a[r][c];
      for (int j = 0; j < 2 * m; ++j) a[r][j] -= f * a[c][j];
    }
  }
  for (int i = 0; i < m; ++i)
    for (int j = 0; j < m; ++j) out[i * m + j] = a[i][m + j];
  return true;
}

__global__ void __launch_bounds__(BI_THREADS)
k_bilu_rows(int m, const int64_t* __restrict__ rows, const int64_t* __restrict__ row_ptr,
            const int32_t* __restrict__ col, const int32_t* __restrict__ ord, const int32_t* __restrict__ nlow,
            double* __restrict__ F, double* __restrict__ Uinv, int* __restrict__ flag) {
  __shared__ double Lb[25];
  const int tid = threadIdx.x, mm = m * m;
  const int64_t i = rows[blockIdx.x];
  const int64_t lo = row_ptr[i];
  const int len = (int)(row_ptr[i + 1] - lo);
  const int32_t* o = ord + lo;
  const int nl = nlow[i];
  for (int q = 0; q < nl; ++q) {
    const int64_t kk = lo + o[q];
    const int64_t k = col[kk];
    if (tid < mm) {
      const int r = tid / m, c = tid % m;
      double sacc = 0.0;
      for (int t = 0; t < m; ++t) sacc = fma(F[kk * mm + r * m + t], Uinv[k * mm + t * m + c], sacc);
      Lb[tid] = sacc;
    }
    __syncthreads();
    if (tid < mm) F[kk * mm + tid] = Lb[tid];
    const int64_t klo = row_ptr[k], khi = row_ptr[k + 1];
    for (int p = q + 1 + tid; p < len; p += BI_THREADS) {
      const int64_t jj = lo + o[p];
      const int32_t j = col[jj];
      int64_t a = klo, b = khi;
      while (a < b) {
        const int64_t mid = (a + b) >> 1;
        if (col[mid] < j) a = mid + 1; else b = mid;
      }
      if (a < khi && col[a] == j) {
        double* dst = F + jj * mm;
        const double* U = F + a * mm;
        for (int r = 0; r < m; ++r)
          for (int c = 0; c < m; ++c) {
            double sacc = dst[r * m + c];
            for (int t = 0; t < m; ++t) sacc = fma(-Lb[r * m + t], U[t * m + c], sacc);
            dst[r * m + c] = sacc;
          }
      }
    }
    __syncthreads();
  }
  if (tid == 0 && !invert_block(m, F + (lo + o[nl]) * mm, Uinv + i * mm)) atomicOr(flag, 1);
}

// BILU(0) factors and elimination orders on the device.
struct BiluTab {
  const int64_t *rows, *row_ptr;
  const int32_t *col, *ord, *nlow;
  const double *F, *Uinv;
};

// One row of the forward (lower) or backward (upper) solve by one warp, in place:
// v_i -= sum_{k before i} L_ik v_k, or v_i = U_ii^-1 (v_i - sum_{j after i} U_ij v_j).
// v is read through L2: other CTAs of the same launch write it in the combined solve.
template <bool FWD>
__device__ __forceinline__ void bilu_row(int m, const BiluTab& B, int64_t i, double* __restrict__ v) {
  const int lane = threadIdx.x & 31, mm = m * m;
  const int64_t lo = B.row_ptr[i];
  const int nl = B.nlow[i];
  const int q0 = FWD ? 0 : nl + 1, q1 = FWD ? nl : (int)(B.row_ptr[i + 1] - lo);
  double acc[5] = {0, 0, 0, 0, 0};
  for (int q = q0 + lane; q < q1; q += 32) {
    const int64_t kk = lo + B.ord[lo + q];
    const double* blk = B.F + kk * mm;
    const double* x = v + (int64_t)B.col[kk] * m;
    double xs[5];
#pragma unroll
    for (int t = 0; t < 5; ++t) xs[t] = t < m ? __ldcg(x + t) : 0.0;
    for (int r = 0; r < m; ++r) {
      double sacc = 0.0;
#pragma unroll
      for (int t = 0; t < 5; ++t)
        if (t < m) sacc = fma(blk[r * m + t], xs[t], sacc);
      acc[r] += sacc;
    }
  }
  for (int r = 0; r < m; ++r)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], off);
  double sv[5];
  for (int t = 0; t < m; ++t) sv[t] = __ldcg(v + i * m + t) - acc[t];
  __syncwarp();
  if (lane < m) {
    double x = sv[lane];
    if (!FWD) {
      x = 0.0;
      for (int t = 0; t < m; ++t) x = fma(B.Uinv[i * mm + lane * m + t], sv[t], x);
    }
    __stcg(v + i * m + lane, x);
  }
}

// Rows of one colour, one warp per row.
template <bool FWD>
__global__ void k_bilu_colour(int m, int64_t nrows, int64_t first, BiluTab B, double* __restrict__ v) {
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w < nrows) bilu_row<FWD>(m, B, B.rows[first + w], v);
}

// ---------------------------------------------------------------- GMRES in one launch
// The solve is a cooperative launch of at most one CTA per SM; its CTAs meet at grid
// barriers, so an Arnoldi step costs three of them instead of a dozen launches and a
// synchronisation with the host (about 100 us a step).  Each CTA owns a contiguous range
// of trace nodes: it forms those rows of K v (one lane per block entry, so that K
// streams in order), preconditions, orthogonalises and normalises
// them; the Hessenberg column, the rotations and the stopping test are formed by every
// CTA from the same sums in the same order, so nothing else is exchanged.  K v is bound
// by the FP64 pipe (one multiply-add per entry of K, two per SM and clock).
// Measured to 1e-12, launch by launch -> one launch (in brackets: a warp per block row, its
// longest row the critical path of every step): 2D p = 2 8 x 8 (768 unknowns, 26 steps)
// 5.04 -> 0.73 ms [0.70], 3D p = 3 6^3 (20,520 unknowns, 112 MB of K, 48 steps) 12.9 -> 3.3
// [5.7], 3D p = 2 16^3 (143,360 unknowns, 72 steps) 31.0 -> 14.3 [20.7]; with BILU(0) 2D
// 3.4 -> 2.5.
constexpr int GK_THREADS = 512, GK_WARPS = GK_THREADS / 32;
constexpr int GK_MIN_ROWS = 8;                    // trace nodes per CTA on small systems
constexpr int GK_BARRIER_POLLS = 1 << 24;

struct GmresArgs {
  int m;
  int64_t T;
  const int64_t* row_ptr;
  const int32_t* col;
  const double *K, *Dinv, *R;
  double *dU, *V, *w;           // V [restart + 1][T m], w [T m]
  double* part;                 // partial sums [2][CTA][R1], the halves in turn (dot_parts)
  double* out;                  // iterations, relative residual
  unsigned* sync;               // [0] barrier count, [1] abort
  int restart, max_iter;
  double rtol;
  int colours;                  // BILU(0): number of colours, 0 = block Jacobi
  const int64_t* cptr;
  BiluTab B;
};
constexpr int GK_R1 = IEDG_MAX_RESTART + 1;

struct GmresShared {
  double red[GK_WARPS][GK_R1 + 1];
  double h1[GK_R1], h2[GK_R1];
  double H[GK_R1][IEDG_MAX_RESTART], cs[IEDG_MAX_RESTART], sn[IEDG_MAX_RESTART], g[GK_R1], y[IEDG_MAX_RESTART];
  double psum[GK_WARPS][2][5];            // K x: the warps' shares of rows they do not hold alone
  int prow[GK_WARPS][2];
  double nrm2, rel, hn, scale;
  int done, abort, again;
};

// Barrier over the grid (all CTAs resident: cooperative launch) in two halves, so that
// work of one thread can hide behind the wait.  Bounded: a CTA that gives up sets the
// abort flag, which ends every CTA's wait.  barrier_wait returns false on abort.
__device__ __forceinline__ void barrier_arrive(const GmresArgs& a) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(a.sync, 1u);
  }
}
__device__ __forceinline__ bool barrier_wait(const GmresArgs& a, GmresShared& sh, unsigned& round) {
  if (threadIdx.x == 0) {
    ++round;
    const unsigned want = round * gridDim.x;
    int polls = 0, ab = 0;
    unsigned seen;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.sync) : "memory");
      if ((int)(seen - want) >= 0) break;
      if ((++polls & 1023) == 0) ab = *(volatile unsigned*)(a.sync + 1) != 0;
    } while (!ab && polls < GK_BARRIER_POLLS);
    if ((int)(seen - want) < 0) { atomicExch(a.sync + 1, 1u); ab = 1; }
    sh.abort = ab;
  }
  __syncthreads();
  return sh.abort == 0;
}
__device__ __forceinline__ bool grid_barrier(const GmresArgs& a, GmresShared& sh, unsigned& round) {
  barrier_arrive(a);
  return barrier_wait(a, sh, round);
}

// Sums over the grid go through a.part: every CTA writes its own row (dot_parts), meets
// the others at a grid barrier and reads all rows (sum_parts).  Successive sums alternate
// between two halves (`turn`, the same in every thread of every CTA).  A row is written again
// two sums later, so there is always the barrier of the sum in between: a CTA arrives there
// only after it has read all rows of the earlier sum, and no CTA writes before all have
// arrived.  (With one half, a CTA that leaves the barrier first could overwrite its row with
// the next sum's while another has yet to read it.)
__device__ __forceinline__ double* part_rows(const GmresArgs& a, unsigned turn) {
  return a.part + (int64_t)(turn & 1u) * kGmresMaxCtas * GK_R1;
}

// out[v] = sum over the grid of part[cta][v], v < nv, in CTA order within a warp's share;
// the same in every CTA.  Ends the sum: the next one takes the other half.
__device__ __forceinline__ void sum_parts(const GmresArgs& a, GmresShared& sh, int nv, double* out, unsigned& turn) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double* part = part_rows(a, turn++);
  for (int v0 = 0; v0 < nv; v0 += 32) {
    double s = 0.0;
    if (v0 + lane < nv)
#pragma unroll 10
      for (int c = warp; c < (int)gridDim.x; c += GK_WARPS) s += __ldcg(part + (int64_t)c * GK_R1 + v0 + lane);
    if (v0 + lane < nv) sh.red[warp][v0 + lane] = s;
  }
  __syncthreads();
  if (threadIdx.x < nv) {
    double s = 0.0;
    const int nw = min(GK_WARPS, (int)gridDim.x);
    for (int k = 0; k < nw; ++k) s += sh.red[k][threadIdx.x];
    out[threadIdx.x] = s;
  }
  __syncthreads();
}

// part[this CTA][v] = V[v] . w over the CTA's unknowns [i0, i1), v < nv: a warp per vector,
// or several where there are more warps than vectors.
__device__ __forceinline__ void dot_parts(const GmresArgs& a, GmresShared& sh, int nv, const double* V, int64_t n,
                                          const double* w, int64_t i0, int64_t i1, unsigned turn) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int segs = nv < GK_WARPS ? GK_WARPS / nv : 1;
  for (int it = warp; it < nv * segs; it += GK_WARPS) {
    const int v = it / segs, sg = it % segs;
    const double* x = V + (int64_t)v * n;
    double s = 0.0;
#pragma unroll 4
    for (int64_t i = i0 + sg * 32 + lane; i < i1; i += 32 * segs) s = fma(x[i], w[i], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) sh.red[sg][v] = s;
  }
  __syncthreads();
  if (threadIdx.x < nv) {
    double s = 0.0;
    for (int k = 0; k < segs; ++k) s += sh.red[k][threadIdx.x];
    __stcg(part_rows(a, turn) + (int64_t)blockIdx.x * GK_R1 + threadIdx.x, s);
  }
}

// Rows [t0, t1) of y = K x, or b - K x; x read through L2 (other CTAs wrote it).  The CTA's
// blocks of K, consecutive in memory, are split evenly over its warps (a block row's
// length varies with the elements at its node); rows that cross warps are summed in warp
// order at the end.  A lane per block entry (two blocks at a time where M = 4; the spare
// lanes repeat others), the column indices read 32 at a time, GK_UN blocks of K and x
// requested together.  Ends with the CTA's threads in step.
constexpr int GK_UN = 16;
template <int M>
__device__ __forceinline__ void spmv_rows_m(const GmresArgs& a, GmresShared& sh, const double* __restrict__ x,
                                            double* __restrict__ y, const double* __restrict__ b, int64_t t0, int64_t t1) {
  constexpr int MM = M * M, PER = 32 / MM;                 // blocks per warp step
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sub = PER > 1 ? (lane / MM) % PER : 0, e = lane % MM, k = e % M;
  if (lane < 2) sh.prow[warp][lane] = -1;
  __syncwarp();
  const int64_t q0 = a.row_ptr[t0], nq = a.row_ptr[t1] - q0;
  int64_t q = q0 + nq * warp / GK_WARPS;
  const int64_t qb = q0 + nq * (warp + 1) / GK_WARPS, qa = q;
  int64_t t = t0;
  if (q < qb) {                                            // row of block q
    int64_t lo = t0, hi = t1;                              // last row that starts at or before q
    while (hi - lo > 1) {
      const int64_t mid = (lo + hi) >> 1;
      if (a.row_ptr[mid] <= q) lo = mid;
      else hi = mid;
    }
    t = lo;
  }
  for (; q < qb; ++t) {
    const int64_t rend = a.row_ptr[t + 1], end = min(rend, qb);
    double acc = 0.0;
    for (int64_t base = q; base < end; base += 32) {
      const int nblk = (int)min((int64_t)32, end - base);
      const int xc = lane < nblk ? a.col[base + lane] * M : 0;
      const double* kb = a.K + base * MM + sub * MM + e;
      const double* xk = x + k;
      int u0 = 0;
      for (; u0 + GK_UN * PER <= nblk; u0 += GK_UN * PER) {
        double kv[GK_UN], xv[GK_UN];
#pragma unroll
        for (int u = 0; u < GK_UN; ++u) {
          kv[u] = kb[(u0 + u * PER) * MM];
          xv[u] = __ldcg(xk + __shfl_sync(0xffffffffu, xc, u0 + u * PER + sub));
        }
#pragma unroll
        for (int u = 0; u < GK_UN; ++u) acc = fma(kv[u], xv[u], acc);
      }
      for (; u0 < nblk; u0 += 4 * PER) {
        double kv[4], xv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int p = u0 + u * PER + sub;
          const int xo = __shfl_sync(0xffffffffu, xc, p & 31);
          const bool on = p < nblk;
          kv[u] = on ? kb[(u0 + u * PER) * MM] : 0.0;
          xv[u] = on ? __ldcg(xk + xo) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) acc = fma(kv[u], xv[u], acc);
      }
    }
    if (PER == 2) acc += __shfl_down_sync(0xffffffffu, acc, 16);
    double s = 0.0;
#pragma unroll
    for (int kk = 0; kk < M; ++kk) s += __shfl_sync(0xffffffffu, acc, (lane < M ? lane * M : 0) + kk);
    if (q == a.row_ptr[t] && end == rend) {
      if (lane < M) y[t * M + lane] = b ? b[t * M + lane] - s : s;
    } else {
      const int slot = q == qa ? 0 : 1;
      if (lane < M) sh.psum[warp][slot][lane] = s;
      if (lane == 0) sh.prow[warp][slot] = (int)(t - t0);
    }
    q = end;
  }
  __syncthreads();
  if (threadIdx.x < M) {                                   // rows shared by warps, in warp order
    int cur = -1;
    double v = 0.0;
    for (int w = 0; w < 2 * GK_WARPS; ++w) {
      const int r = sh.prow[w >> 1][w & 1];
      if (r < 0) continue;
      if (r != cur) {
        if (cur >= 0) y[(t0 + cur) * M + threadIdx.x] = b ? b[(t0 + cur) * M + threadIdx.x] - v : v;
        cur = r;
        v = 0.0;
      }
      v += sh.psum[w >> 1][w & 1][threadIdx.x];
    }
    if (cur >= 0) y[(t0 + cur) * M + threadIdx.x] = b ? b[(t0 + cur) * M + threadIdx.x] - v : v;
  }
  __syncthreads();
}
__device__ __forceinline__ void spmv_rows(const GmresArgs& a, GmresShared& sh, const double* x, double* y,
                                          const double* b, int64_t t0, int64_t t1) {
  if (a.m == 5) spmv_rows_m<5>(a, sh, x, y, b, t0, t1);
  else spmv_rows_m<4>(a, sh, x, y, b, t0, t1);
}

// z = M^-1 y on the CTA's rows: block Jacobi, or BILU(0) in place on all rows of y (other
// CTAs work on this one's rows: barriers inside, y read through L2) and then copied.
__device__ __forceinline__ bool precondition(const GmresArgs& a, GmresShared& sh, double* y, double* z, int64_t t0,
                                             int64_t t1, unsigned& round) {
  const int tid = threadIdx.x, m = a.m;
  const int64_t i0 = t0 * m, i1 = t1 * m;
  if (a.colours == 0) {
    for (int64_t i = i0 + tid; i < i1; i += GK_THREADS) {
      const int64_t t = i / m;
      double s = 0.0;
#pragma unroll
      for (int k = 0; k < 5; ++k)
        if (k < m) s = fma(a.Dinv[i * m + k], y[t * m + k], s);
      z[i] = s;
    }
    __syncthreads();
    return true;
  }
  const int64_t w0 = (int64_t)blockIdx.x * GK_WARPS + (tid >> 5), nw = (int64_t)gridDim.x * GK_WARPS;
  if (!grid_barrier(a, sh, round)) return false;
  for (int c = 0; c < a.colours; ++c) {
    for (int64_t r = a.cptr[c] + w0; r < a.cptr[c + 1]; r += nw) bilu_row<true>(a.m, a.B, a.B.rows[r], y);
    if (!grid_barrier(a, sh, round)) return false;
  }
  for (int c = a.colours - 1; c >= 0; --c) {
    for (int64_t r = a.cptr[c] + w0; r < a.cptr[c + 1]; r += nw) bilu_row<false>(a.m, a.B, a.B.rows[r], y);
    if (!grid_barrier(a, sh, round)) return false;
  }
  for (int64_t i = i0 + tid; i < i1; i += GK_THREADS) z[i] = __ldcg(y + i);
  __syncthreads();
  return true;
}

// First trace node of CTA b: the rows are split by blocks of K.
__device__ __forceinline__ int64_t first_row(const GmresArgs& a, int b) {
  const int64_t want = a.row_ptr[a.T] * b / (int)gridDim.x;
  int64_t lo = 0, hi = a.T;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (a.row_ptr[mid] < want) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

__global__ void __launch_bounds__(GK_THREADS, 1) k_gmres(GmresArgs a) {
  __shared__ GmresShared sh;
  const int tid = threadIdx.x;
  const int m = a.m;
  const int64_t n = a.T * m;
  const int64_t t0 = first_row(a, blockIdx.x), t1 = blockIdx.x + 1 == gridDim.x ? a.T : first_row(a, blockIdx.x + 1);
  const int64_t i0 = t0 * m, i1 = t1 * m;
  unsigned round = 0, turn = 0;
  // x0 = 0, r0 = M^-1 R
  for (int64_t i = i0 + tid; i < i1; i += GK_THREADS) {
    a.dU[i] = 0.0;
    a.w[i] = a.R[i];
  }
  __syncthreads();
  // own rows of x <- s (x - sum_{v < nv} h[v] V_v)
  auto subtract = [&](int nv, const double* h, double* x, double s) {
    for (int64_t i = i0 + tid; i < i1; i += GK_THREADS) {
      double t = x[i];
#pragma unroll 8
      for (int v = 0; v < nv; ++v) t = fma(-h[v], a.V[(int64_t)v * n + i], t);
      x[i] = s * t;
    }
  };
  int total = 0;
  double beta0 = 0.0, relres = 0.0;
  bool first = true, alive = true;
  while (alive) {
    if (!first) spmv_rows(a, sh, a.dU, a.w, a.R, t0, t1);
    if (!(alive = precondition(a, sh, a.w, a.V, t0, t1, round))) break;
    dot_parts(a, sh, 1, a.V, n, a.V, i0, i1, turn);
    if (!(alive = grid_barrier(a, sh, round))) break;
    sum_parts(a, sh, 1, sh.h1, turn);
    const double beta = sqrt(sh.h1[0]);
    if (first) {
      beta0 = beta;
      relres = beta0 > 0.0 ? 1.0 : 0.0;
    } else {
      relres = beta / beta0;
    }
    first = false;
    if (!(beta0 > 0.0) || total >= a.max_iter || relres <= a.rtol) break;
    {
      const double s = beta > 0.0 ? 1.0 / beta : 0.0;
      for (int64_t i = i0 + tid; i < i1; i += GK_THREADS) a.V[i] *= s;
      for (int i = tid; i < GK_R1; i += GK_THREADS) sh.g[i] = i == 0 ? beta : 0.0;
    }
    if (!(alive = grid_barrier(a, sh, round))) break;
    // Hessenberg column c: earlier rotations applied, a new one formed, g rotated,
    // |g_{c+1}| / beta0 the residual estimate
    auto givens = [&](int c) {
      const double hn = sh.hn;
      double a0 = sh.h1[0] + sh.h2[0];
      for (int i = 0; i < c; ++i) {
        const double a1 = sh.h1[i + 1] + sh.h2[i + 1];
        sh.H[i][c] = sh.cs[i] * a0 + sh.sn[i] * a1;
        a0 = -sh.sn[i] * a0 + sh.cs[i] * a1;
      }
      const double r = hypot(a0, hn);
      const double cc = r > 0.0 ? a0 / r : 1.0, sn = r > 0.0 ? hn / r : 0.0;
      sh.cs[c] = cc;
      sh.sn[c] = sn;
      sh.H[c][c] = r;
      const double gc = sh.g[c];
      sh.g[c + 1] = -sn * gc;
      sh.g[c] = cc * gc;
      sh.rel = fabs(sh.g[c + 1]) / beta0;
      sh.done = (sh.rel <= a.rtol || hn == 0.0) ? 1 : 0;
    };
    int j = 0;
    for (;;) {
      // one thread closes step j - 1 while the others start on K v_j: the stopping test
      // costs at most a product that is not used
      const bool more = j < a.restart && total < a.max_iter;
      if (j > 0 && tid >= GK_THREADS - 32) {
        if (tid == GK_THREADS - 32) givens(j - 1);
        __syncwarp();
      }
      if (more) spmv_rows(a, sh, a.V + (int64_t)j * n, a.w, nullptr, t0, t1);
      else __syncthreads();
      if (j > 0) {
        relres = sh.rel;
        if (sh.done || !more) break;
      }
      double* vn = a.V + (int64_t)(j + 1) * n;
      if (!(alive = precondition(a, sh, a.w, vn, t0, t1, round))) break;
      // iterated classical Gram-Schmidt: two passes, the second with |w|^2 beside the
      // products (V_{j+1} is w itself), which gives the norm of the orthogonalised
      // vector, |w|^2 - |h2|^2, without another barrier
      dot_parts(a, sh, j + 1, a.V, n, vn, i0, i1, turn);
      if (!(alive = grid_barrier(a, sh, round))) break;
      sum_parts(a, sh, j + 1, sh.h1, turn);
      subtract(j + 1, sh.h1, vn, 1.0);
      __syncthreads();
      dot_parts(a, sh, j + 2, a.V, n, vn, i0, i1, turn);
      if (!(alive = grid_barrier(a, sh, round))) break;
      sum_parts(a, sh, j + 2, sh.h2, turn);
      if (tid < 32) {        // one warp: square roots and divisions would load the FP64 pipe
        double q = 0.0;
        for (int v = tid; v <= j; v += 32) q = fma(sh.h2[v], sh.h2[v], q);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
        const double w2 = sh.h2[j + 1], hn2 = w2 - q;
        if (tid == 0) {
          // a second pass that still removes much of w would cancel here: sum again then
          sh.again = hn2 < 0.25 * w2;
          const double r = hn2 > 0.0 ? 1.0 / sqrt(hn2) : 0.0;
          sh.hn = hn2 * r;
          sh.scale = sh.again ? 1.0 : r;
        }
      }
      __syncthreads();
      subtract(j + 1, sh.h2, vn, sh.scale);
      if (sh.again) {
        __syncthreads();
        dot_parts(a, sh, 1, vn, n, vn, i0, i1, turn);
        if (!(alive = grid_barrier(a, sh, round))) break;
        sum_parts(a, sh, 1, &sh.nrm2, turn);
        if (tid == 0) {
          sh.hn = sqrt(sh.nrm2);
          sh.scale = sh.nrm2 > 0.0 ? 1.0 / sh.hn : 0.0;
        }
        __syncthreads();
        const double s = sh.scale;
        for (int64_t i = i0 + tid; i < i1; i += GK_THREADS) vn[i] *= s;
      }
      if (!(alive = grid_barrier(a, sh, round))) break;   // v_{j+1} complete
      ++j;
      ++total;
    }
    if (!alive) break;
    // y = H(0:j, 0:j)^-1 g (upper triangular, column by column), x += V y
    if (tid < 32) {
      for (int i = j - 1; i >= 0; --i) {
        const double yi = sh.g[i] / sh.H[i][i];
        __syncwarp();
        for (int k = tid; k < i; k += 32) sh.g[k] = fma(-sh.H[k][i], yi, sh.g[k]);
        if (tid == 0) sh.y[i] = yi;
        __syncwarp();
      }
    }
    __syncthreads();
    for (int64_t i = i0 + tid; i < i1; i += GK_THREADS) {
      double s = a.dU[i];
      for (int v = 0; v < j; ++v) s = fma(sh.y[v], a.V[(int64_t)v * n + i], s);
      a.dU[i] = s;
    }
    if (!(total < a.max_iter && relres > a.rtol)) break;
    if (!(alive = grid_barrier(a, sh, round))) break;     // x complete before K x
  }
  if (blockIdx.x == 0 && tid == 0) {
    a.out[0] = (double)total;
    a.out[1] = relres;
  }
}

}  // namespace

#define SV_TRY(call)                                                                       \
  do {                                                                                     \
    cudaError_t e_ = (call);                                                               \
    if (e_ != cudaSuccess) {                                                               \
      M->err = std::string("iedg_trace_solve: ") + #call + ": " + cudaGetErrorString(e_); \
      return IEDG_ERR_CUDA;                                                                \
    }                                                                                      \
  } while (0)

// Colouring and elimination orders of the trace pattern (host, once per handle).
static int bilu_setup(iedg_mesh* M, cudaStream_t st) {
  if (M->brows) return IEDG_OK;
  const int64_t T = M->T, nnzb = M->nnzb;
  std::vector<int64_t> rp(T + 1);
  std::vector<int32_t> col(nnzb);
  SV_TRY(cudaMemcpyAsync(rp.data(), M->row_ptr, (T + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  SV_TRY(cudaMemcpyAsync(col.data(), M->col, nnzb * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  SV_TRY(cudaStreamSynchronize(st));
  // greedy colouring in index order
  std::vector<int32_t> color(T, -1), mark;
  int32_t ncol = 0;
  for (int64_t t = 0; t < T; ++t) {
    mark.assign(ncol + 1, 0);
    for (int64_t k = rp[t]; k < rp[t + 1]; ++k)
      if (col[k] < t) mark[color[col[k]]] = 1;
    int32_t c = 0;
    while (mark[c]) ++c;
    color[t] = c;
    if (c + 1 > ncol) ncol = c + 1;
  }
  // rows sorted by (colour, index); rank = position in that order
  std::vector<int64_t> rows(T), cnt(ncol + 1, 0), rank(T);
  for (int64_t t = 0; t < T; ++t) cnt[color[t] + 1]++;
  for (int32_t c = 0; c < ncol; ++c) cnt[c + 1] += cnt[c];
  M->bcptr = cnt;
  {
    std::vector<int64_t> fill(cnt.begin(), cnt.end() - 1);
    for (int64_t t = 0; t < T; ++t) rows[fill[color[t]]++] = t;
  }
  for (int64_t r = 0; r < T; ++r) rank[rows[r]] = r;
  // per row: entries in elimination order, and how many come before the row
  std::vector<int32_t> ord(nnzb), nlow(T);
  for (int64_t t = 0; t < T; ++t) {
    const int64_t lo = rp[t];
    const int32_t len = (int32_t)(rp[t + 1] - lo);
    int32_t* o = ord.data() + lo;
    for (int32_t q = 0; q < len; ++q) o[q] = q;
    std::sort(o, o + len, [&](int32_t a, int32_t b) { return rank[col[lo + a]] < rank[col[lo + b]]; });
    int32_t nl = 0;
    while (nl < len && rank[col[lo + o[nl]]] < rank[t]) ++nl;
    nlow[t] = nl;
  }
  auto put = [&](auto** dst, const auto& h) -> cudaError_t {
    using E = typename std::remove_const<typename std::remove_reference<decltype(h[0])>::type>::type;
    E* d = nullptr;
    cudaError_t e = cudaMalloc((void**)&d, std::max<size_t>(h.size(), 1) * sizeof(E));
    if (e != cudaSuccess) return e;
    M->allocs.push_back(d);
    M->ws_bytes += (int64_t)(h.size() * sizeof(E));
    *dst = d;
    return cudaMemcpyAsync(d, h.data(), h.size() * sizeof(E), cudaMemcpyHostToDevice, st);
  };
  SV_TRY(put(&M->bcptr_dev, cnt));
  SV_TRY(put(&M->brows, rows));
  SV_TRY(put(&M->bord, ord));
  SV_TRY(put(&M->bnlow, nlow));
  SV_TRY(cudaStreamSynchronize(st));
  M->bcolor = color;
  return IEDG_OK;
}

static int bilu_factor(iedg_mesh* M, const double* K, double* F, cudaStream_t st) {
  int rc = bilu_setup(M, st);
  if (rc != IEDG_OK) return rc;
  const int m = M->dm.m;
  if (F != K) SV_TRY(cudaMemcpyAsync(F, K, (size_t)M->nnzb * m * m * sizeof(double), cudaMemcpyDeviceToDevice, st));
  SV_TRY(cudaMemsetAsync(M->dev_flag, 0, sizeof(int), st));
  for (size_t c = 0; c + 1 < M->bcptr.size(); ++c) {
    const int64_t nr = M->bcptr[c + 1] - M->bcptr[c];
    if (nr == 0) continue;
    SV_TRY((k_bilu_rows<<<(unsigned)nr, BI_THREADS, 0, st>>>(m, M->brows + M->bcptr[c], M->row_ptr, M->col, M->bord,
                                                             M->bnlow, F, M->dinv, M->dev_flag),
            cudaGetLastError()));
  }
  int flag = 0;
  SV_TRY(cudaMemcpyAsync(&flag, M->dev_flag, sizeof(int), cudaMemcpyDeviceToHost, st));
  SV_TRY(cudaStreamSynchronize(st));
  if (flag) {
    M->err = "BILU(0): singular pivot block";
    return IEDG_ERR_INVALID_ARG;
  }
  return IEDG_OK;
}

// v <- U^-1 L^-1 v, colour by colour (one launch per colour and sweep: a single-block
// form of all colours was measured slower, one SM's bandwidth for the whole factor)
static cudaError_t bilu_apply(iedg_mesh* M, const double* F, double* v, cudaStream_t st) {
  const int m = M->dm.m;
  const size_t nc = M->bcptr.size() - 1;
  const BiluTab B{M->brows, M->row_ptr, M->col, M->bord, M->bnlow, F, M->dinv};
  auto blocks = [](int64_t nr) { return (unsigned)((nr * 32 + SV_THREADS - 1) / SV_THREADS); };
  for (size_t c = 0; c < nc; ++c) {
    const int64_t nr = M->bcptr[c + 1] - M->bcptr[c];
    if (nr > 0) k_bilu_colour<true><<<blocks(nr), SV_THREADS, 0, st>>>(m, nr, M->bcptr[c], B, v);
  }
  for (size_t c = nc; c-- > 0;) {
    const int64_t nr = M->bcptr[c + 1] - M->bcptr[c];
    if (nr > 0) k_bilu_colour<false><<<blocks(nr), SV_THREADS, 0, st>>>(m, nr, M->bcptr[c], B, v);
  }
  return cudaGetLastError();
}

extern "C" int iedg_set_trace_precond(iedg_mesh* M, int32_t kind) {
  if (!M) return IEDG_ERR_INVALID_ARG;
  if (kind != IEDG_PREC_BLOCK_JACOBI && kind != IEDG_PREC_BILU0) {
    M->err = "iedg_set_trace_precond: unknown preconditioner";
    return IEDG_ERR_INVALID_ARG;
  }
  M->prec_kind = kind;
  return IEDG_OK;
}

extern "C" int iedg_bilu0_factor(iedg_mesh* M, const double* K, double* F, void* stream) {
  if (!M || !K || !F) {
    if (M) M->err = "iedg_bilu0_factor: null argument";
    return IEDG_ERR_INVALID_ARG;
  }
  return bilu_factor(M, K, F, (cudaStream_t)stream);
}

extern "C" int iedg_bilu0_apply(iedg_mesh* M, const double* F, const double* r, double* x, void* stream) {
  if (!M || !F || !r || !x) {
    if (M) M->err = "iedg_bilu0_apply: null argument";
    return IEDG_ERR_INVALID_ARG;
  }
  if (!M->brows) {
    M->err = "iedg_bilu0_apply: no factorisation on this handle";
    return IEDG_ERR_NOT_ASSEMBLED;
  }
  cudaStream_t st = (cudaStream_t)stream;
  if (x != r) SV_TRY(cudaMemcpyAsync(x, r, (size_t)M->T * M->dm.m * sizeof(double), cudaMemcpyDeviceToDevice, st));
  SV_TRY(bilu_apply(M, F, x, st));
  return IEDG_OK;
}

extern "C" int iedg_trace_colors(iedg_mesh* M, int32_t* colors) {
  if (!M || !colors) return IEDG_ERR_INVALID_ARG;
  int rc = bilu_setup(M, 0);
  if (rc != IEDG_OK) return rc;
  std::memcpy(colors, M->bcolor.data(), M->bcolor.size() * sizeof(int32_t));
  return IEDG_OK;
}

extern "C" int iedg_trace_solve(iedg_mesh* M, const double* K, const double* R, double* dU, int32_t restart,
                                int32_t max_iter, double rtol, int32_t* iterations, double* rel_residual,
                                void* stream) {
  if (!M || !K || !R || !dU) {
    if (M) M->err = "iedg_trace_solve: null argument";
    return IEDG_ERR_INVALID_ARG;
  }
  if (restart < 1 || restart > IEDG_MAX_RESTART || max_iter < 1 || !(rtol > 0.0)) {
    M->err = "iedg_trace_solve: restart must be 1..IEDG_MAX_RESTART, max_iter >= 1, rtol > 0";
    return IEDG_ERR_INVALID_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const int m = M->dm.m;
  const int64_t T = M->T, n = T * m;
  const bool bilu = M->prec_kind == IEDG_PREC_BILU0;
  if (bilu) {
    if (!M->bf) {
      double* f = nullptr;
      SV_TRY(cudaMalloc(&f, (size_t)M->nnzb * m * m * sizeof(double)));
      M->allocs.push_back(f);
      M->ws_bytes += (int64_t)M->nnzb * m * m * sizeof(double);
      M->bf = f;
    }
    int rc = bilu_factor(M, K, M->bf, st);
    if (rc != IEDG_OK) return rc;
  }
  SV_TRY(cudaMemsetAsync(M->dev_flag, 0, sizeof(int), st));
  if (!bilu)
    SV_TRY((k_diag_inv<<<(unsigned)((T + 127) / 128), 128, 0, st>>>(m, T, M->row_ptr, M->col, K, M->dinv, M->dev_flag),
            cudaGetLastError()));
  // result scalars and the barrier's two words sit behind the partial sums
  double* out = M->kpart + 2 * (int64_t)GK_R1 * kGmresMaxCtas;
  unsigned* sync = reinterpret_cast<unsigned*>(out + 4);
  SV_TRY(cudaMemsetAsync(out, 0, 8 * sizeof(double), st));
  GmresArgs a{m, T, M->row_ptr, M->col, K, M->dinv, R, dU, M->kry, M->kry + (int64_t)GK_R1 * n, M->kpart, out, sync,
              restart, max_iter, rtol, bilu ? (int)M->bcptr.size() - 1 : 0, M->bcptr_dev,
              BiluTab{M->brows, M->row_ptr, M->col, M->bord, M->bnlow, M->bf, M->dinv}};
  // one CTA per SM at most (a co-resident grid with the fewest partial sums), fewer on small systems
  int dev = 0, sms = 0;
  SV_TRY(cudaGetDevice(&dev));
  SV_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t g = std::min<int64_t>(std::min<int64_t>(sms, kGmresMaxCtas), std::max<int64_t>(1, T / GK_MIN_ROWS));
  void* args[] = {&a};
  SV_TRY(cudaLaunchCooperativeKernel((const void*)k_gmres, dim3((unsigned)g), dim3(GK_THREADS), args, 0, st));
  double res[5] = {0, 0, 0, 0, 0};
  int flag = 0;
  SV_TRY(cudaMemcpyAsync(res, out, sizeof(res), cudaMemcpyDeviceToHost, st));
  SV_TRY(cudaMemcpyAsync(&flag, M->dev_flag, sizeof(int), cudaMemcpyDeviceToHost, st));
  SV_TRY(cudaStreamSynchronize(st));
  if (flag && !bilu) {
    M->err = "iedg_trace_solve: singular diagonal block of K";
    return IEDG_ERR_INVALID_ARG;
  }
  unsigned words[2];
  std::memcpy(words, &res[4], sizeof(words));
  if (words[1]) {
    M->err = "iedg_trace_solve: the grid barrier gave up";
    return IEDG_ERR_CUDA;
  }
  if (iterations) *iterations = (int32_t)res[0];
  if (rel_residual) *rel_residual = res[1];
  return IEDG_OK;
}
