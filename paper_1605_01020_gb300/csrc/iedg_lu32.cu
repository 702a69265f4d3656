// FP32 partial LU of the bordered element matrices (mixed path): every update on FFMA, or
// with the Schur complement deferred to one GEMM on the tensor cores (TF32 in two parts,
// TF32 or BF16 operands).  Every trailing update on the tensor cores: iedg_lu32_mma.cu.
//
// Same algorithm and pivot rule as lu_element (iedg_assemble.cu).  What the refinement
// reads is written back: the full panels (L, in the row order of their own step) and the
// pivot rows.
//
// Per 32-column panel: the u-rows are factored in shared memory (column-major, two barriers
// a column: the pass that applies one column's multipliers finds the next column's
// pivot), the trace rows, which hold no pivots, are then solved against U11 one row per
// thread without a barrier, the trailing columns are permuted and solved against L11 one
// column per thread, and A22 -= L21 U12 runs over 64 x 128 tiles (128 threads; 8 x 8
// registers each, four 16-byte shared loads per 64 multiply-adds), L21 and U12 staged per
// tile.  Each entry takes its 32 multiply-adds of a panel in the same order in every
// form, so results do not depend on the tiling.
// CTAs of 128 threads, four per SM where shared memory allows: the column steps of one
// element's panel are latency, which the other elements' updates fill.
// Measured, the form before (panels over all rows with three barriers a column, 256
// threads, 4 x 8 tiles) -> this one: p = 3, 4096 elements 34.5 -> 31.8 ms; p = 4, 210 elements
// 20.4 -> 16.6 ms; TF32 Schur operands, p = 3, 504 elements 6.09 -> 5.87 ms.  Issue slots 40 %
// busy, 23 MB of DRAM traffic per element: the trailing block passes through L2 once per
// panel.
#include <cuda_bf16.h>

#include "iedg_internal.cuh"
#include "iedg_lu_common.cuh"
#include "iedg_tc.cuh"

namespace iedg {
namespace {

constexpr int L32_NB = 32;
constexpr int L32_TH = 128;          // threads of the FFMA form (the tensor-core forms: LU_THREADS)
constexpr int L32_TN = 128;          // columns of an update tile
constexpr int L32_LPAD = 4;          // padding of a staged column of L21

// rows of an update tile: 16 threads across, 8 rows each
constexpr int l32_rows(int th) { return th / 16 * 8; }
__host__ __device__ inline int l32_stride(int nu) { return nu | 1; }

inline size_t l32_smem(const Dims& dm, int th) {
  const size_t panel = (size_t)L32_NB * l32_stride(dm.nu), tile = (size_t)L32_NB * (L32_TN + l32_rows(th) + L32_LPAD);
  return sizeof(float) * (panel > tile ? panel : tile);
}

struct Lu32Shared {
  int piv[L32_NB];
  float inv[L32_NB];                 // reciprocal pivots of the panel
  int perm[LU_MAX_NU];               // net row permutation of the panel's interchanges
  float rv[LU_THREADS / 32];
  int ri[LU_THREADS / 32];
  int sing;
};

// Panel columns over the u-rows, P column-major (column j at P + j PR).
template <int TH>
__device__ __forceinline__ void lu32_panel(Lu32Shared& sh, float* P, int PR, int prow, int nb, int kb, int* pivots,
                                           int& nonfin) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int j = 0; j < nb; ++j) {
    float best = -1.f;
    int bi = j;
    auto candidate = [&](float x, int r) {
      const float v = fabsf(x);
      nonfin |= !(v <= 3.402823466e38f);
      if (v > best) { best = v; bi = r; }
    };
    if (j == 0) {
      for (int r = tid; r < prow; r += TH) candidate(P[r], r);
    } else {
      const float inv = sh.inv[j - 1];
      const float* piv_row = P + (j - 1);
      for (int r = j + tid; r < prow; r += TH) {
        float* row = P + r;
        const float l = row[(j - 1) * PR] * inv;
        row[(j - 1) * PR] = l;
        const float v = fmaf(-l, piv_row[j * PR], row[j * PR]);
        row[j * PR] = v;
        candidate(v, r);
#pragma unroll 4
        for (int c = j + 1; c < nb; ++c) row[c * PR] = fmaf(-l, piv_row[c * PR], row[c * PR]);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
    }
    if (lane == 0) { sh.rv[warp] = best; sh.ri[warp] = bi; }
    __syncthreads();
    if (warp == 0) {
      float bv = sh.rv[0];
      int pr = sh.ri[0];
      for (int w = 1; w < TH / 32; ++w)
        if (sh.rv[w] > bv || (sh.rv[w] == bv && sh.ri[w] < pr)) { bv = sh.rv[w]; pr = sh.ri[w]; }
      if (!(bv > 0.f)) pr = j;
      const float pv = P[pr + j * PR];
      __syncwarp();
      if (lane == 0) {
        if (!(bv > 0.f)) sh.sing = 1;
        sh.inv[j] = pv != 0.f ? 1.f / pv : 0.f;
        sh.piv[j] = pr;
        pivots[kb + j] = kb + pr;
        if (pr != j) { const int t = sh.perm[j]; sh.perm[j] = sh.perm[pr]; sh.perm[pr] = t; }
      }
      if (pr != j) {
        const float t = P[j + lane * PR];
        P[j + lane * PR] = P[pr + lane * PR];
        P[pr + lane * PR] = t;
      }
    }
    __syncthreads();
  }
  const float inv = sh.inv[nb - 1];      // the last column's multipliers
  for (int r = nb + tid; r < prow; r += TH) P[r + (nb - 1) * PR] *= inv;
  __syncthreads();
}

// A[r][c] -= sum_j L[r][j] U[j][c] over rows [r_lo, r_hi), cols [c_lo, c_hi), L = columns
// kb .. kb+nb-1 and U = rows kb .. kb+nb-1 of A.  `check`: `bad` collects non-finite results.
template <int TH>
__device__ __forceinline__ void lu32_update(float* __restrict__ A, int ld, float* __restrict__ sm, int kb, int nb,
                                            int r_lo, int r_hi, int c_lo, int c_hi, int vlim, bool check, int& bad) {
  constexpr int RT = l32_rows(TH), LS = RT + L32_LPAD;
  float* Us = sm;                               // [32][128]
  float* Ls = sm + L32_NB * L32_TN;             // [32][LS]
  const int tid = threadIdx.x, tc = tid & 15, tr = tid >> 4;
  const bool aligned = ((c_lo | kb) & 3) == 0;
  for (int cc = c_lo; cc < c_hi; cc += L32_TN) {
    __syncthreads();                            // the previous tile is done with Us
    for (int q = tid; q < L32_NB * (L32_TN / 4); q += TH) {
      const int j = q / (L32_TN / 4), c = 4 * (q % (L32_TN / 4));
      const float* src = A + (int64_t)(kb + j) * ld + cc + c;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j < nb) {
        if (aligned && cc + c + 4 <= vlim) {
          v = *reinterpret_cast<const float4*>(src);
        } else {
          if (cc + c < c_hi) v.x = src[0];
          if (cc + c + 1 < c_hi) v.y = src[1];
          if (cc + c + 2 < c_hi) v.z = src[2];
          if (cc + c + 3 < c_hi) v.w = src[3];
        }
      }
      *reinterpret_cast<float4*>(Us + j * L32_TN + c) = v;
    }
    for (int rb = r_lo; rb < r_hi; rb += RT) {
      if (rb != r_lo) __syncthreads();          // the previous row block is done with Ls
      for (int q = tid; q < RT * (L32_NB / 4); q += TH) {
        // lane -> 8 rows x 4 pieces of 4 columns: two-way conflicts at most
        const int w = q >> 5, l = q & 31, r = 8 * (w >> 1) + (l & 7), j = 4 * ((l >> 3) + 4 * (w & 1));
        const float* src = A + (int64_t)(rb + r) * ld + kb + j;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (rb + r < r_hi) {
          if (j + 4 <= nb) {
            v = *reinterpret_cast<const float4*>(src);       // kb and ld are multiples of 4
          } else {
            if (j < nb) v.x = src[0];
            if (j + 1 < nb) v.y = src[1];
            if (j + 2 < nb) v.z = src[2];
          }
        }
        Ls[j * LS + r] = v.x;
        Ls[(j + 1) * LS + r] = v.y;
        Ls[(j + 2) * LS + r] = v.z;
        Ls[(j + 3) * LS + r] = v.w;
      }
      // this thread's 8 rows x (4 + 4) columns (an L2 prefetch of the next row block's lines, kept
      // inside the matrix, made it slower: p = 3 31.8 -> 32.9 ms, p = 4 16.6 -> 18.4)
      float acc[8][8];
      const int ca = cc + 4 * tc, cb = ca + 64;
      const bool va = aligned && ca + 4 <= vlim, vb = aligned && cb + 4 <= vlim;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = rb + 8 * tr + i;
        const float* src = A + (int64_t)r * ld;
        float4 p = make_float4(0.f, 0.f, 0.f, 0.f), q = p;
        if (r < r_hi) {
          if (va) {
            p = *reinterpret_cast<const float4*>(src + ca);
          } else {
            if (ca < c_hi) p.x = src[ca];
            if (ca + 1 < c_hi) p.y = src[ca + 1];
            if (ca + 2 < c_hi) p.z = src[ca + 2];
            if (ca + 3 < c_hi) p.w = src[ca + 3];
          }
          if (vb) {
            q = *reinterpret_cast<const float4*>(src + cb);
          } else {
            if (cb < c_hi) q.x = src[cb];
            if (cb + 1 < c_hi) q.y = src[cb + 1];
            if (cb + 2 < c_hi) q.z = src[cb + 2];
            if (cb + 3 < c_hi) q.w = src[cb + 3];
          }
        }
        acc[i][0] = p.x; acc[i][1] = p.y; acc[i][2] = p.z; acc[i][3] = p.w;
        acc[i][4] = q.x; acc[i][5] = q.y; acc[i][6] = q.z; acc[i][7] = q.w;
      }
      __syncthreads();
      if (cc + 64 >= c_hi) {               // nothing in the right half of the tile
#pragma unroll 4
        for (int j = 0; j < nb; ++j) {
          const float4 l0 = *reinterpret_cast<const float4*>(Ls + j * LS + 8 * tr);
          const float4 l1 = *reinterpret_cast<const float4*>(Ls + j * LS + 8 * tr + 4);
          const float4 u0 = *reinterpret_cast<const float4*>(Us + j * L32_TN + 4 * tc);
          const float lv[8] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
          const float uv[4] = {u0.x, u0.y, u0.z, u0.w};
#pragma unroll
          for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(-lv[a], uv[b], acc[a][b]);
        }
      } else
#pragma unroll 4
      for (int j = 0; j < nb; ++j) {
        const float4 l0 = *reinterpret_cast<const float4*>(Ls + j * LS + 8 * tr);
        const float4 l1 = *reinterpret_cast<const float4*>(Ls + j * LS + 8 * tr + 4);
        const float4 u0 = *reinterpret_cast<const float4*>(Us + j * L32_TN + 4 * tc);
        const float4 u1 = *reinterpret_cast<const float4*>(Us + j * L32_TN + 64 + 4 * tc);
        const float lv[8] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
        const float uv[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int b = 0; b < 8; ++b) acc[a][b] = fmaf(-lv[a], uv[b], acc[a][b]);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = rb + 8 * tr + i;
        float* dst = A + (int64_t)r * ld;
        if (r >= r_hi) break;
        if (va) {
          *reinterpret_cast<float4*>(dst + ca) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        } else {
#pragma unroll
          for (int b = 0; b < 4; ++b)
            if (ca + b < c_hi) dst[ca + b] = acc[i][b];
        }
        if (vb) {
          *reinterpret_cast<float4*>(dst + cb) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
        } else {
#pragma unroll
          for (int b = 0; b < 4; ++b)
            if (cb + b < c_hi) dst[cb + b] = acc[i][4 + b];
        }
        if (check)
#pragma unroll
          for (int b = 0; b < 4; ++b)
            bad |= (ca + b < c_hi && !isfinite(acc[i][b])) || (cb + b < c_hi && !isfinite(acc[i][4 + b]));
      }
    }
  }
  __syncthreads();
}

// Deferred Schur complement on the tensor cores: [K | R] = [D | G] - W [Z | z] for rows
// [nu, n) and columns [nu, n], W = A[nu:n, 0:nu] (the eliminated trace rows, L21 of
// every panel) and Z = A[0:nu, nu:n] (U12 of every panel), so K accumulates over the
// whole K = nu in TMEM and the trace block is read and written once.  128 x 64 output
// tiles, K chunks of 32 in two operand stages so that one chunk is staged while the
// tensor core works on the other; one thread issues the MMAs, completion through
// per-stage mbarriers with bounded waits; the epilogue reads TMEM with all eight warps.
// Operand forms (KIND): kSchurFp32 = TF32 high and low parts, three products (hi hi +
// hi lo + lo hi, FP32 accuracy, 48 KB stages); kSchurTf32 = one product of the operands
// rounded to TF32 (24 KB); kSchurBf16 = one product of BF16 operands (12 KB).  All
// accumulate in FP32.
constexpr int TC_TM = 128, TC_TN = 64, TC_KC = 32;
constexpr int TC_STAGE_BYTES = 2 * TC_TM * TC_KC * 4 + 2 * TC_TN * TC_KC * 4;   // 48 KB, the largest form

template <int KIND>
struct SchurForm {
  static constexpr int EB = KIND == kSchurBf16 ? 2 : 4;          // bytes per operand value
  static constexpr int PARTS = KIND == kSchurFp32 ? 2 : 1;       // hi (+ lo)
  static constexpr int A_BYTES = TC_TM * TC_KC * EB, B_BYTES = TC_TN * TC_KC * EB;
  static constexpr int SBO = TC_KC * EB / 16 * 128;               // 8-row group stride
  __device__ static uint32_t off(int row, int k) { return EB == 4 ? tc::core_off32(row, k) : tc::core_off16(row, k); }
  // value v at (row, k) of the A (b = false) or B operand tile
  __device__ static void put(char* stage, bool b, int row, int k, float v) {
    char* base = stage + (b ? PARTS * A_BYTES : 0);
    const uint32_t o = off(row, k);
    if constexpr (KIND == kSchurFp32) {
      float hi, lo;
      tc::split_tf32(v, hi, lo);
      *reinterpret_cast<float*>(base + o) = hi;
      *reinterpret_cast<float*>(base + (b ? B_BYTES : A_BYTES) + o) = lo;
    } else if constexpr (KIND == kSchurTf32) {
      *reinterpret_cast<float*>(base + o) = tc::round_tf32(v);
    } else {
      *reinterpret_cast<__nv_bfloat16*>(base + o) = __float2bfloat16_rn(v);
    }
  }
};

template <int KIND>
__device__ __forceinline__ void schur_stage(const float* __restrict__ A, int ld, int n, int nu, int ncol, int rt,
                                            int ct, int kc, char* stage) {
  using F = SchurForm<KIND>;
  const int tid = threadIdx.x;
  // A operand: W rows rt .. rt+127, K columns kc .. kc+31 (k fastest: coalesced rows)
  for (int idx = tid; idx < TC_TM * TC_KC; idx += LU_THREADS) {
    const int mm = idx >> 5, k = idx & 31;
    const int r = rt + mm, c = kc + k;
    F::put(stage, false, mm, k, (r < n && c < nu) ? A[(int64_t)r * ld + c] : 0.f);
  }
  // B operand (N x K, K-major): Z rows kc .. kc+31, columns ct .. ct+63 (column fastest)
  for (int idx = tid; idx < TC_TN * TC_KC; idx += LU_THREADS) {
    const int k = idx >> 6, nn = idx & 63;
    const int r = kc + k, c = ct + nn;
    F::put(stage, true, nn, k, (r < nu && c < ncol) ? A[(int64_t)r * ld + c] : 0.f);
  }
}

template <int KIND>
__device__ __forceinline__ void schur_issue(uint32_t tmem, const char* stage, bool first) {
  using F = SchurForm<KIND>;
  const uint32_t aH = tc::smem_u32(stage), aL = aH + F::A_BYTES;
  const uint32_t bH = aH + F::PARTS * F::A_BYTES, bL = bH + F::B_BYTES;
  // one instruction covers 32 bytes of K (8 TF32 or 16 BF16 values): two core matrices
#pragma unroll
  for (int st = 0; st < TC_KC * F::EB / 32; ++st) {
    const uint32_t ko = st * 256, acc = (first && st == 0) ? 0u : 1u;
    if constexpr (KIND == kSchurBf16) {
      constexpr uint32_t IDESC = tc::idesc_bf16(TC_TM, TC_TN);
      tc::mma_bf16(tmem, tc::desc_kmajor(aH + ko, 128, F::SBO), tc::desc_kmajor(bH + ko, 128, F::SBO), IDESC, acc);
    } else {
      constexpr uint32_t IDESC = tc::idesc_tf32(TC_TM, TC_TN);
      tc::mma_tf32(tmem, tc::desc_kmajor(aH + ko, 128, F::SBO), tc::desc_kmajor(bH + ko, 128, F::SBO), IDESC, acc);
      if constexpr (KIND == kSchurFp32) {
        tc::mma_tf32(tmem, tc::desc_kmajor(aH + ko, 128, F::SBO), tc::desc_kmajor(bL + ko, 128, F::SBO), IDESC, 1);
        tc::mma_tf32(tmem, tc::desc_kmajor(aL + ko, 128, F::SBO), tc::desc_kmajor(bH + ko, 128, F::SBO), IDESC, 1);
      }
    }
  }
}

// Bounded wait on stage b's barrier by every thread; the outcome is made uniform.
// (A wait that ran out leaves the phase where it was, so the drain can wait for it.)
__device__ __forceinline__ bool schur_wait(TcState* tcs, int b) {
  const bool ok = __syncthreads_and(tc::mbar_wait(tcs->mbar + b, tcs->phase[b], tcs->limit));
  if (ok) { tcs->phase[b] ^= 1u; tcs->pending[b] = 0; }
  else tcs->failed = 1;
  return ok;
}

template <int KIND>
__device__ void schur_tc(float* __restrict__ A, int ld, int n, int nu, char* smem, TcState* tcs) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ncol = n + 1;
  const int nk = (nu + TC_KC - 1) / TC_KC;
  const int q = warp & 3, h = warp >> 2;
  for (int rt = nu; rt < n && !tcs->failed; rt += TC_TM) {
    for (int ct = nu; ct < ncol && !tcs->failed; ct += TC_TN) {
      schur_stage<KIND>(A, ld, n, nu, ncol, rt, ct, 0, smem);
      tc::fence_proxy_async();
      __syncthreads();
      tc::fence_after_sync();
      for (int c = 0; c < nk; ++c) {
        const int b = c & 1;
        if (tid == 0) {
          schur_issue<KIND>(tcs->tmem, smem + b * TC_STAGE_BYTES, c == 0);
          tc::mma_commit(tcs->mbar + b);
        }
        tcs->pending[b] = 1;
        if (c + 1 < nk) {
          // the other stage was last read by the MMAs of chunk c - 1
          if (c >= 1 && !schur_wait(tcs, b ^ 1)) break;
          schur_stage<KIND>(A, ld, n, nu, ncol, rt, ct, (c + 1) * TC_KC, smem + (b ^ 1) * TC_STAGE_BYTES);
          tc::fence_proxy_async();
          __syncthreads();
          tc::fence_after_sync();
        }
      }
      if (tcs->failed) break;
      // the two commits not waited for yet: chunks nk - 2 and nk - 1
      if (nk >= 2 && !schur_wait(tcs, (nk - 2) & 1)) break;
      if (!schur_wait(tcs, (nk - 1) & 1)) break;
      tc::fence_after_sync();
      // epilogue: warp (q, h) owns rows 32 q .. 32 q + 31 and columns 32 h .. 32 h + 31
      const int row = rt + 32 * q + lane;
#pragma unroll 1
      for (int c8 = 0; c8 < 4; ++c8) {
        const int c0 = 32 * h + 8 * c8;
        float pv8[8];
        tc::tmem_ld8(tcs->tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c0, pv8);
        if (row >= n || ct + c0 >= ncol) continue;
        float* dst = A + (int64_t)row * ld + ct + c0;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (ct + c0 + j < ncol) dst[j] -= pv8[j];
      }
      tc::fence_before_sync();
      __syncthreads();
    }
  }
}

template <int TH, bool TC, int KIND = kSchurFp32>
__device__ __forceinline__ void lu32_element(Lu32Shared& sh, const LuElem& el, float* __restrict__ S,
                                             int8_t* __restrict__ status, int* __restrict__ pivots, const int64_t e,
                                             TcState* tcs) {
  extern __shared__ __align__(16) unsigned char smraw[];
  float* P = reinterpret_cast<float*>(smraw);          // [NB][PR] column-major panel; update tiles
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = el.n, nu = el.nu, ld = el.ld, ncol = n + 1, PR = l32_stride(nu);
  float* A = S + el.off;
  int nonfin = 0, bad = 0;              // a pivot candidate / the Schur complement is NaN or infinite
  if (tid == 0) sh.sing = 0;
  for (int kb = 0; kb < nu; kb += L32_NB) {
    const int nb = min(L32_NB, nu - kb), prow = nu - kb;
    for (int r = warp; r < prow; r += TH / 32)
      P[r + lane * PR] = lane < nb ? A[(int64_t)(kb + r) * ld + kb + lane] : 0.f;
    for (int r = tid; r < prow; r += TH) sh.perm[r] = r;
    __syncthreads();
    lu32_panel<TH>(sh, P, PR, prow, nb, kb, pivots + el.poff, nonfin);
    // u-rows of the panel back (U11, L11, L21)
    for (int r = warp; r < prow; r += TH / 32)
      if (lane < nb) A[(int64_t)(kb + r) * ld + kb + lane] = P[r + lane * PR];
    // trace rows of L21, x U11 = a: one thread per row
    for (int r = nu + tid; r < n; r += TH) {
      float* row = A + (int64_t)r * ld + kb;
      float x[L32_NB];
#pragma unroll
      for (int j = 0; j < L32_NB; j += 4) {
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        if (j + 4 <= nb) {
          t = *reinterpret_cast<const float4*>(row + j);
        } else {
          if (j < nb) t.x = row[j];
          if (j + 1 < nb) t.y = row[j + 1];
          if (j + 2 < nb) t.z = row[j + 2];
        }
        x[j] = t.x; x[j + 1] = t.y; x[j + 2] = t.z; x[j + 3] = t.w;
      }
#pragma unroll
      for (int j = 0; j < L32_NB; ++j) {
        if (j >= nb) break;
        x[j] *= sh.inv[j];
#pragma unroll
        for (int c = j + 1; c < L32_NB; ++c) x[c] = fmaf(-x[j], P[j + c * PR], x[c]);
      }
#pragma unroll
      for (int j = 0; j < L32_NB; j += 4) {
        if (j + 4 <= nb) {
          *reinterpret_cast<float4*>(row + j) = make_float4(x[j], x[j + 1], x[j + 2], x[j + 3]);
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (j + q < nb) row[j + q] = x[j + q];
        }
      }
    }
    // trailing columns: row interchanges, then U12 = L11^-1 A12.  The panel's
    // interchanges, applied in order, leave row r holding the original row perm[r]; the
    // rows below the panel that change are among the pivot rows piv[j] >= nb, and they
    // receive original rows above nb.  Each column gathers its new top rows first
    // (independent loads), then moves the displaced rows, then stores the top rows.
    for (int c = kb + nb + tid; c < ncol; c += TH) {
      float x[L32_NB];
#pragma unroll
      for (int j = 0; j < L32_NB; ++j) x[j] = j < nb ? A[(int64_t)(kb + sh.perm[j]) * ld + c] : 0.f;
#pragma unroll
      for (int j0 = 0; j0 < L32_NB; j0 += 8) {
        float y[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int r = j0 + j < nb ? sh.piv[j0 + j] : 0;
          y[j] = (j0 + j < nb && r >= nb && sh.perm[r] != r) ? A[(int64_t)(kb + sh.perm[r]) * ld + c] : 0.f;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int r = j0 + j < nb ? sh.piv[j0 + j] : 0;
          if (j0 + j < nb && r >= nb && sh.perm[r] != r) A[(int64_t)(kb + r) * ld + c] = y[j];
        }
      }
#pragma unroll
      for (int j = 0; j < L32_NB; ++j) {
        if (j >= nb) break;
#pragma unroll
        for (int i = j + 1; i < L32_NB; ++i) x[i] = fmaf(-P[i + j * PR], x[j], x[i]);
        A[(int64_t)(kb + j) * ld + c] = x[j];
      }
    }
    __syncthreads();
    const int r0 = kb + nb;
    if constexpr (TC) {
      // deferred Schur complement: the u-columns of every row and the trace columns of
      // the u-rows are updated now (the next panels and U12 need them); the trace block
      // of the trace rows receives all panels at once on the tensor cores below
      lu32_update<TH>(A, ld, P, kb, nb, r0, n, r0, nu, nu, false, bad);
      lu32_update<TH>(A, ld, P, kb, nb, r0, nu, nu, ncol, ld, false, bad);
    } else {
      // A22 -= L21 U12, rows [kb+nb, n), cols [kb+nb, n]
      lu32_update<TH>(A, ld, P, kb, nb, r0, n, r0, ncol, ld, r0 == nu, bad);
    }
  }
  if constexpr (TC) {
    __syncthreads();
    schur_tc<KIND>(A, ld, n, nu, reinterpret_cast<char*>(smraw), tcs);     // the panel buffer is free now
    __syncthreads();
    bad = 0;
    for (int idx = tid; idx < (n - nu) * (ncol - nu); idx += TH) {
      const int r = nu + idx / (ncol - nu), c = nu + idx % (ncol - nu);
      if (!isfinite(A[(int64_t)r * ld + c])) bad = 1;
    }
  }
  bad = __syncthreads_or(bad);
  nonfin = __syncthreads_or(nonfin);
  if (tid == 0) {
    if (TC && tcs->failed) status[e] = IEDG_ELEM_TIMEOUT;
    else status[e] = nonfin ? IEDG_ELEM_NONFINITE
                            : (sh.sing ? IEDG_ELEM_SINGULAR : (bad ? IEDG_ELEM_NONFINITE : IEDG_ELEM_OK));
  }
}

__global__ void __launch_bounds__(L32_TH, 4)
k_lu32(Dims dm, LuDesc lud, float* __restrict__ S, int8_t* __restrict__ status, int* __restrict__ pivots,
       int64_t* queue, int64_t E) {
  __shared__ Lu32Shared sh;
  int64_t e;
  for (int64_t it = 0; next_element(queue, E, it, lud.order, &e); ++it)
    lu32_element<L32_TH, false>(sh, lu_elem(dm, lud, e), S, status, pivots, e, nullptr);
}

// Tensor-core form: TMEM (128 columns) and the completion barrier are set up once per
// CTA; a CTA whose completion wait ran out stops taking elements, waits once more
// (bounded) for its MMAs, and frees its TMEM.
template <int KIND>
__global__ void __launch_bounds__(LU_THREADS, 2)
k_lu32_tc(Dims dm, LuDesc lud, float* __restrict__ S, int8_t* __restrict__ status, int* __restrict__ pivots,
          int64_t* queue, int64_t E, int* err, int wait_limit) {
  __shared__ Lu32Shared sh;
  __shared__ uint32_t tmem_base;
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ TcState tcs;
  const int tid = threadIdx.x, warp = tid >> 5;
  if (warp == 0) {
    tc::tmem_alloc(&tmem_base, TC_TN);
    tc::tmem_relinquish();
  }
  if (tid == 0) {
    tc::mbar_init(&mbar[0], 1);
    tc::mbar_init(&mbar[1], 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (tid == 0) {
    tcs.tmem = tmem_base;
    tcs.mbar = mbar;
    tcs.phase[0] = 0;
    tcs.phase[1] = 0;
    tcs.failed = 0;
    tcs.limit = wait_limit;
    tcs.pending[0] = 0;
    tcs.pending[1] = 0;
  }
  __syncthreads();
  // each thread keeps its own copy of the phases; the shared copy is only the start
  TcState mine = tcs;
  int64_t e;
  int64_t it = 0;
  for (; next_element(queue, E, it, lud.order, &e); ++it) {
    lu32_element<LU_THREADS, true, KIND>(sh, lu_elem(dm, lud, e), S, status, pivots, e, &mine);
    if (__syncthreads_or(mine.failed)) {
      if (tid == 0) atomicOr(err, 1);
      tc_drain(mine);     // MMAs still in flight finish before the TMEM is freed
      ++it;
      break;
    }
  }
  // after a failed wait this CTA factors nothing more: the elements it still takes from
  // the queue are flagged, so no element is left unfactored with an OK status
  if (mine.failed)
    for (; next_element(queue, E, it, lud.order, &e); ++it)
      if (tid == 0) status[e] = IEDG_ELEM_TIMEOUT;
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tmem_base, TC_TN);
}

}  // namespace

// FP32 partial LU with the Schur complement on the tensor cores in operand form KIND.
template <int KIND>
static cudaError_t lu32_tc(iedg_mesh* M, cudaStream_t st) {
  // panel and update tiles during the factorisation; the two operand stages of the Schur GEMM
  // reuse the same buffer afterwards
  size_t smem = l32_smem(M->dm, LU_THREADS);
  if (smem < 2 * (size_t)TC_STAGE_BYTES) smem = 2 * (size_t)TC_STAGE_BYTES;
  cudaError_t err = cudaFuncSetAttribute(k_lu32_tc<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  unsigned grid = (unsigned)M->E;
  int64_t* queue = nullptr;
  if (M->sched.lu_persistent) {
    err = persistent_grid(k_lu32_tc<KIND>, smem, M->E, &grid);
    if (err == cudaSuccess) err = cudaMemsetAsync(M->queue, 0, sizeof(int64_t), st);
    if (err != cudaSuccess) return err;
    queue = M->queue;
  }
  k_lu32_tc<KIND><<<grid, LU_THREADS, smem, st>>>(M->dm, M->lud, M->S32, M->status, M->piv, queue, M->E, M->dev_flag,
                                                   tc_wait_limit(M));
  return cudaGetLastError();
}

cudaError_t launch_lu32(iedg_mesh* M, cudaStream_t st) {
  if (M->schur_in == kSchurTf32) return lu32_tc<kSchurTf32>(M, st);
  if (M->schur_in == kSchurBf16) return lu32_tc<kSchurBf16>(M, st);
  if (M->sched.lu_tensor) return lu32_tc<kSchurFp32>(M, st);
  const size_t smem = l32_smem(M->dm, L32_TH);
  cudaError_t err = cudaFuncSetAttribute(k_lu32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  unsigned grid = (unsigned)M->E;
  int64_t* queue = nullptr;
  if (M->sched.lu_persistent) {
    err = persistent_grid(k_lu32, smem, M->E, &grid, 64, L32_TH);
    if (err == cudaSuccess) err = cudaMemsetAsync(M->queue, 0, sizeof(int64_t), st);
    if (err != cudaSuccess) return err;
    queue = M->queue;
  }
  k_lu32<<<grid, L32_TH, smem, st>>>(M->dm, M->lud, M->S32, M->status, M->piv, queue, M->E);
  return cudaGetLastError();
}

}  // namespace iedg
