// FP64 element matrices of hexahedra (degree 2..4, p + 2 points per direction) with the
// contractions over the points on the tensor cores, by splitting the FP64 operands into
// 8-bit digits.
//
// For equation i and unknown k the u-rows are products of tables that all elements share
// and of the pair's right operands at the volume and face points (iedg_assemble.cu),
//   sum_{g,r} Dxi_r[g][a] W_r[g][col] + sum_fp PhiF[fp][a] V[fp][col] + alpha delta_ik M,
//   W_r[g][b] = cu_ikr(g) Phi[g][b] - sum_l cq_iklr(g) Gl_l(g)[b],  V likewise,
// and the trace rows of uniform meshes are the face parts of the boundary nodes' u-rows.
// Sum-factorised on the FP64 pipe the contractions are two thirds of the assembly's
// multiply-adds (two per SM and clock on GB300).  Here only W and V are formed in FP64; the
// contractions, dense, run as exact integer products of digits (iedg_digits.cuh):
//   * the MMA's A operand (128 TMEM lanes) is the table, lane a = test function a; its
//     digits are laid out once per handle in operand order, 16 values of K (32 KB) at a
//     time, and stream through a ring of bulk copies;
//   * the B operand is W (V) for 32 columns of the element, which may belong to several
//     pairs: the digits t are stacked, so that digit s of the table meets all digits t <=
//     7 - s in one instruction (see k_lu64_tc);
//   * a column's scale is the exponent of its largest |W| (|V|), which k_w_exp finds in FP32
//     beforehand, so W is converted as it is formed;
//   * FP32 level sums stay exact (below 2^24) over a window of chunks, checked for the
//     tables' own digits when they are laid out; then the levels are joined in 96-bit
//     integers, rounded once to FP64 and added to the element matrix.
// Warps: 8 form and convert W and read the accumulators, one issues the MMAs, one the
// copies; they meet at mbarriers, all waits bounded.  Two CTAs per SM, so that one's
// conversion and results overlap the other's FP64.
// Meshes with mixed orders have trace bases of their own: there the face terms come from
// k_assemble_sf first and this kernel adds the volume terms.
// Accuracy.  An entry's error is about 2^-58 of (largest table value of its row) (largest |W| of
// its column), then one FP64 rounding; FP64 sums round every term.  Errors of the element
// matrix and, through an exact elimination, of K against 80-bit arithmetic (numpy model, FP64
// sums | this kernel, median entry): p = 3, Re 2.5e5, cubes 1.4e-16 7.4e-16 | 1.0e-16 3.3e-16;
// p = 3, Re 1e4, cells 1 : 50 1.6e-16 1.2e-15 | 1.2e-16 3.9e-16; p = 3, Re 0.1, M 0.01, cells
// 1 : 1000 1.8e-16 1.8e-12 | 1.1e-16 1.1e-12 (with the bound from separate maxima as scale
// 4.5e-15 1.4e-14, 9.3e-15 2.5e-14, 4.8e-15 2.4e-11).
// Measured, all elements, sum-factorised on the FP64 pipe -> this form (k_coef_exp, k_w_exp,
// k_assemble_dg): 3D p = 3, 4096 elements 135.4 -> 100.6 ms; p = 2, 2002 elements 14.0 ->
// 13.1 ms; p = 4, 210 elements 32.8 -> 18.8 ms; orders 2, 3, 4 mixed, 324 elements 25.6 ->
// 17.4 ms.  Counters at p = 3: FP64 pipe 50 % busy, tensor pipe 26 %, 7.9 TB/s from L2, two
// thirds of it the tables.
#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "iedg_digits.cuh"
#include "iedg_internal.cuh"
#include "iedg_tc.cuh"

namespace iedg {
namespace {

constexpr int DG_BUILD = 256, DG_THREADS = DG_BUILD + 64;   // build warps, MMA warp, copy warp
constexpr int DG_COLS = 32, DG_GP = 16;                     // columns of a tile, K of a step
constexpr int DG_SLICE = 128 * DG_GP * 2;                   // one digit of the table's 128 lanes
constexpr int DG_STEP_A = dig::S * DG_SLICE;                // 32 KB
constexpr int DG_RING = 2;
constexpr int DG_STEP_B = dig::S * DG_COLS * DG_GP * 2;     // 8 KB
constexpr size_t DG_SMEM = (size_t)DG_RING * DG_STEP_A + 3 * DG_STEP_B + 128;

// byte offset of (row, k) in a K = 16 operand slice (core matrices of 8 x 8 BF16)
__host__ __device__ __forceinline__ uint32_t dg_off(int row, int k) {
  return (uint32_t)((row >> 3) * 256 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}
// a chunk is three steps: 48 face points, or 16 volume points in the three directions
__host__ __device__ constexpr int dg_face_chunks(int Nfp) { return (Nfp + 3 * DG_GP - 1) / (3 * DG_GP); }
__host__ __device__ constexpr int dg_vol_chunks(int Nq) { return (Nq + DG_GP - 1) / DG_GP; }

struct DgShared {
  // table stage filled / read, right operands staged / read, accumulators complete / read, end
  uint64_t full[DG_RING], empty[DG_RING], bfull, bempty, dfull, dread, drain;
  uint32_t tmem;
  int failed;
  int scol[DG_COLS];        // column of the bordered matrix, -1 = none
  int sblk[DG_COLS];        // equation component
  int mcol[DG_COLS];        // column of the mass matrix of diagonal pairs, -1 = none
  int sexp[2][DG_COLS];     // scales (biased exponents): face, volume
};

struct DgArgs {
  AsmTab<double> tb;
  RefTables ref;
  const int16_t* ecoef;           // [E][25][9] largest exponents of cu, cq_l; fuh, fq_l; S_ik (lambda)
  const int16_t* elift;           // [E][6][Np + Nb] largest exponents of the columns of Gl, Hl: volume, face
  int16_t* ew;                    // [slot][25][2][Np + Nb] exponents of the columns of V, W (k_w_exp)
  const double* rhs64;            // mixed handles: FP64 right-hand sides
  double* S;
  double alpha;
  TraceTab tt;
  const int64_t* elist;           // list form: element of each slot
  int64_t n_el;
  int wait_limit;                 // polls of a wait before it gives up
};

template <int NP1, bool MIX>
__global__ void __launch_bounds__(DG_THREADS, 2) k_assemble_dg(Dims dm, DgArgs a, int tiles) {
  constexpr int NQ1 = NP1 + 1, Np = NP1 * NP1 * NP1, Nq = NQ1 * NQ1 * NQ1, Nfp = 6 * NQ1 * NQ1, m2 = 25;
  constexpr int NbU = Np - (NP1 - 2) * (NP1 - 2) * (NP1 - 2);
  constexpr int NFC = dg_face_chunks(Nfp), NVC = dg_vol_chunks(Nq);
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned char* ring = smraw + ((128u - (tc::smem_u32(smraw) & 127u)) & 127u);
  unsigned char* bbuf = ring + DG_RING * DG_STEP_A;
  __shared__ __align__(8) DgShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int NbT = MIX ? dm.Nb : NbU;
  if (warp == 8) {
    tc::tmem_alloc(&sh.tmem, 256);
    tc::tmem_relinquish();
  }
  if (tid == 0) {
    for (int i = 0; i < DG_RING; ++i) { tc::mbar_init(&sh.full[i], 1); tc::mbar_init(&sh.empty[i], 1); }
    tc::mbar_init(&sh.bfull, DG_BUILD / 32);
    tc::mbar_init(&sh.bempty, 1);
    tc::mbar_init(&sh.dfull, 1);
    tc::mbar_init(&sh.dread, DG_BUILD / 32);
    tc::mbar_init(&sh.drain, 1);
    sh.failed = 0;
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = sh.tmem;
  volatile int* failed = &sh.failed;
  // All roles meet at mbarriers and every wait on them is bounded.  Once one has run out the
  // others poll only once: the copies and the MMAs stop (no stage is overwritten), what is in
  // flight is waited for, and the build warps go through the tiles that are left writing NaN.
  // Arrivals then no longer match the waits, which costs nothing: nobody waits for them.
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    // (the flag is read only when the first poll, the usual case, did not do)
    bool ok = a.wait_limit > 0 && tc::mbar_wait(bar, parity & 1u, 1);
    if (!ok) ok = tc::mbar_wait(bar, parity & 1u, *failed ? 1 : a.wait_limit);
    if (!ok) *failed = 1;
    return ok;
  };
  // element, trace slots, first column and chunk range of tile `id`; false: nothing to do
  const int ch0 = MIX ? NFC : 0;
  auto tile_of = [&](int64_t id, int64_t& slot, int64_t& e, int& nb, int& c0, int& ch1) {
    slot = id / tiles;
    c0 = (int)(id % tiles) * DG_COLS;
    e = a.elist ? a.elist[slot] : slot;
    nb = (MIX && e >= 0) ? a.tt.nb[e] : NbU;
    const bool vol = c0 < 17 * (Np + nb) + 8 * Np;
    ch1 = vol ? NFC + NVC : NFC;
    return e >= 0 && ch0 < ch1 && c0 < m2 * (Np + nb);
  };
  // the chunks' windows: all face chunks, then Vwindow volume chunks at a time
  auto window_end = [&](int ch, int ch1) {
    return ch + 1 == ch1 || ch + 1 == NFC || (ch >= NFC && (ch + 1 - NFC) % a.ref.Vwindow == 0);
  };
  const int64_t total = a.n_el * tiles;

  if (warp == 9) {
    // ---- copies of the tables
    if (lane == 0) {
      uint32_t q = 0;
      for (int64_t id = blockIdx.x; id < total && !*failed; id += gridDim.x) {
        int64_t slot, e;
        int nb, c0, ch1;
        if (!tile_of(id, slot, e, nb, c0, ch1)) continue;
        for (int s = 3 * ch0; s < 3 * ch1; ++s, ++q) {
          const uint32_t st = q % DG_RING;
          if (q >= DG_RING && !wait(&sh.empty[st], q / DG_RING - 1)) break;
          tc::mbar_expect_tx(&sh.full[st], DG_STEP_A);
          tc::bulk_g2s(ring + st * DG_STEP_A, a.ref.Vdig + (size_t)s * DG_STEP_A, DG_STEP_A, &sh.full[st]);
        }
      }
      // nothing in flight at exit
      for (uint32_t k = q > DG_RING ? q - DG_RING : 0; k < q; ++k)
        tc::mbar_wait(&sh.full[k % DG_RING], (k / DG_RING) & 1u, kTcWaitLimit);
    }
  } else if (warp == 8) {
    // ---- MMAs
    if (lane == 0) {
      const uint64_t da0 = tc::desc_kmajor(tc::smem_u32(ring), 128, 256);
      const uint64_t db0 = tc::desc_kmajor(tc::smem_u32(bbuf), 128, 256);
      uint32_t q = 0, nch = 0, nwin = 0;
      bool start = true;
      for (int64_t id = blockIdx.x; id < total && !*failed; id += gridDim.x) {
        int64_t slot, e;
        int nb, c0, ch1;
        if (!tile_of(id, slot, e, nb, c0, ch1)) continue;
        for (int ch = ch0; ch < ch1; ++ch, ++nch) {
          bool ok = !start || nwin == 0 || wait(&sh.dread, nwin - 1);   // accumulators read
          ok = ok && wait(&sh.bfull, nch) && !*failed;                  // W of this chunk staged
          const bool end = window_end(ch, ch1);
          for (int r = 0; r < 3; ++r, ++q) {
            const uint32_t st = q % DG_RING;
            ok = ok && wait(&sh.full[st], q / DG_RING);
            if (!ok) break;
            tc::fence_after_sync();
#pragma unroll
            for (int s = 0; s < dig::S; ++s)
              tc::mma_bf16(tmem + (uint32_t)(s * DG_COLS), da0 + (uint64_t)((st * DG_STEP_A + s * DG_SLICE) >> 4),
                           db0 + (uint64_t)((r * DG_STEP_B) >> 4), tc::idesc_bf16(128, DG_COLS * (dig::S - s)),
                           (start && r == 0 && s == 0) ? 0u : 1u);
            tc::mma_commit(&sh.empty[st]);
          }
          if (!ok) break;
          tc::mma_commit(&sh.bempty);
          if (end) tc::mma_commit(&sh.dfull);
          nwin += end;
          start = end;
        }
      }
      if (q > 0) {       // no MMA in flight when the TMEM is freed
        tc::mma_commit(&sh.drain);
        tc::mbar_wait(&sh.drain, 0, kTcWaitLimit);
      }
    }
    __syncwarp();
  } else {
    // ---- right operands and results
    const int c = lane, gq = warp;                 // column of the tile, values 2 gq, 2 gq + 1 of every step
    const int qt = warp & 3, h = warp >> 2, row = 32 * qt + lane;
    const int rexpF = a.ref.Vexp[row], rexpV = a.ref.Vexp[128 + row];
    const int srow = (!MIX && row < Np) ? a.ref.slot[row] : -1;      // trace slot of the lane's node
    uint32_t nch = 0, nwin = 0;
    for (int64_t id = blockIdx.x; id < total; id += gridDim.x) {
      int64_t slot, e;
      int nb, c0, ch1;
      if (!tile_of(id, slot, e, nb, c0, ch1)) continue;
      // this thread's column
      const HexCol hc = hex_col(c0 + c, Np, nb);
      const int col = hc.col;
      const bool ucol = hc.u, cq = hc.cq;
      int pair = hc.pair;
      const bool on = pair >= 0;
      if (!on) pair = 0;
      const int pi = pair / 5, pk = pair % 5, gst = ucol ? Np : NbT;
      const size_t ep = (size_t)e * m2 + pair;
      const double* GV = ucol ? a.tb.GlV + (size_t)e * 3 * Nq * Np + col : a.tb.HlV + (size_t)e * 3 * Nq * NbT + col;
      const double* GF = ucol ? a.tb.GlF + (size_t)e * 3 * Nfp * Np + col : a.tb.HlF + (size_t)e * 3 * Nfp * NbT + col;
      const double* jv = a.tb.Jv + ep * (size_t)(12 * Nq);
      const double* jf = a.tb.Jf + ep * (size_t)(4 * Nfp);
      // face coefficient of the basis value: dfhat/duhat, or dfhat/du = lambda I / S_ik
      const double* jfu = !ucol ? jf : (a.tb.Su ? a.tb.Su + ep * Nfp : a.tb.lamw + (size_t)e * Nfp);
      const bool fu = on && (!ucol || a.tb.Su != nullptr || pi == pk);
      const int bcol = ucol ? col : (MIX ? 0 : a.ref.bnode[col]);
      int emF = 0, emV = 0;
      if (on) {
        const int16_t* ew = a.ew + ((size_t)slot * m2 + pair) * 2 * (Np + NbT) + (ucol ? col : Np + col);
        emF = ew[0];
        emV = ew[Np + NbT];
      }
      asm volatile("bar.sync 3, 256;" ::: "memory");          // the last tile's results are written
      if (gq == 0) {
        sh.scol[c] = !on ? -1 : (ucol ? pk * Np + col : dm.nu + pk * nb + col);
        sh.sblk[c] = pi;
        sh.mcol[c] = (on && ucol && pi == pk) ? col : -1;
        sh.sexp[0][c] = dig::scale_of(emF);
        sh.sexp[1][c] = dig::scale_of(emV);
      }
      asm volatile("bar.sync 3, 256;" ::: "memory");
      const int64_t nn = MIX ? (int64_t)dm.nu + 5 * (int64_t)nb : dm.n;
      const int64_t ld = MIX ? a.tt.ldv[e] : dm.ld;
      double* Se = MIX ? a.S + a.tt.soff[e] : a.S + slot * nn * ld;
      if (!MIX && a.rhs64 != nullptr && c0 == 0)
        for (int r = tid; r < nn; r += DG_BUILD) Se[r * ld + nn] = a.rhs64[e * dm.n + r];
      double gl[2][3], phv[2];
      auto fetch = [&](int vc) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int g = vc * DG_GP + 2 * gq + i;
          const bool ok = on && g < Nq;
          phv[i] = (ok && ucol) ? a.tb.Phi[(size_t)g * Np + col] : 0.0;
#pragma unroll
          for (int l = 0; l < 3; ++l) gl[i][l] = (ok && cq) ? GV[((size_t)l * Nq + g) * gst] : 0.0;
        }
      };
      if (MIX) fetch(0);
      for (int ch = ch0; ch < ch1; ++ch, ++nch) {
        double w[3][2];
        const bool face = !MIX && ch < NFC;
        if (face) {
#pragma unroll
          for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const int fp = ch * 3 * DG_GP + r * DG_GP + 2 * gq + i;
              double v = 0.0;
              if (fp < Nfp && fu) v = jfu[fp] * a.tb.PhiF[(size_t)fp * Np + bcol];
              if (fp < Nfp && on && cq) {
#pragma unroll
                for (int l = 0; l < 3; ++l) {
                  const double x = GF[((size_t)l * Nfp + fp) * gst];
                  v = fma(jf[(size_t)(1 + l) * Nfp + fp], ucol ? -x : x, v);
                }
              }
              w[r][i] = v;
            }
        } else {
          const int vc = ch - NFC;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int g = min(vc * DG_GP + 2 * gq + i, Nq - 1);   // past the end: zero factors
#pragma unroll
            for (int r = 0; r < 3; ++r) w[r][i] = ucol ? jv[(size_t)r * Nq + g] * phv[i] : 0.0;
            if (cq) {
#pragma unroll
              for (int l = 0; l < 3; ++l) {
                const double gv = ucol ? -gl[i][l] : gl[i][l];
#pragma unroll
                for (int r = 0; r < 3; ++r) w[r][i] = fma(jv[(size_t)(3 + 3 * l + r) * Nq + g], gv, w[r][i]);
              }
            }
          }
        }
        if (ch + 1 >= NFC && ch + 1 < ch1) fetch(ch + 1 - NFC);
        const int em = face ? emF : emV;
        if (nch == 0 || wait(&sh.bempty, nch - 1)) {            // the MMAs have read the previous chunk
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            const unsigned long long v0 = dig::to_bytes<false>(__double_as_longlong(w[r][0]), em);
            const unsigned long long v1 = dig::to_bytes<false>(__double_as_longlong(w[r][1]), em);
            unsigned char* base = bbuf + r * DG_STEP_B + dg_off(c, 2 * gq);
#pragma unroll
            for (int s = 0; s < dig::S; ++s)
              *reinterpret_cast<uint32_t*>(base + s * (DG_COLS * DG_GP * 2)) =
                  s < 4 ? dig::bf16_pair((uint32_t)(v0 >> 32), (uint32_t)(v1 >> 32), s)
                        : dig::bf16_pair((uint32_t)v0, (uint32_t)v1, s);
          }
        }
        tc::fence_proxy_async();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&sh.bfull);
        if (window_end(ch, ch1)) {
          bool bad = !wait(&sh.dfull, nwin++);
          tc::fence_after_sync();
          if (32 * qt < Np) {
            bad |= *failed != 0;
            const int rexp = face ? rexpF : rexpV;
            const bool init = !MIX && ch < NFC;
#pragma unroll 1
            for (int c4 = 0; c4 < 4; ++c4) {
              const int cb = 16 * h + 4 * c4;
              double* dst[4];
              double s[4];
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const int sc = sh.scol[cb + j];
                dst[j] = (row < Np && sc >= 0) ? Se + ((int64_t)sh.sblk[cb + j] * Np + row) * ld + sc : nullptr;
                s[j] = (!init && dst[j]) ? *dst[j] : 0.0;
                if (init && dst[j] && sh.mcol[cb + j] >= 0)
                  s[j] = a.alpha * a.tb.Mass[((size_t)e * Np + row) * Np + sh.mcol[cb + j]];
              }
              float t[8][4];
              dig::load_levels(tmem + ((uint32_t)(32 * qt) << 16) + (uint32_t)cb, DG_COLS, t);
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                int v[8];
#pragma unroll
                for (int l = 0; l < 8; ++l) v[l] = __float2int_rn(t[l][j]);
                const long long H = (long long)(v[0] * 256 + v[1]) * 65536 + (long long)v[2] * 256 + v[3];
                const long long L = (long long)v[4] * 16777216 + (long long)v[5] * 65536 + (long long)v[6] * 256 + v[7];
                // 62 leading bits of H 2^32 + L
                const int sf = min(32, __clzll((H ^ (H >> 63)) | 1) - 2);
                const long long x = (long long)((unsigned long long)H << sf) + (L >> (32 - sf));
                const unsigned long long sg = (unsigned long long)(x >> 63);
                const unsigned long long mag = ((unsigned long long)x ^ sg) - sg;
                const int lz = __clzll((long long)(mag | 1ull));
                const int ef = rexp + sh.sexp[face ? 0 : 1][cb + j];
                bool odd;
                double r = dig::from_fixed(mag, lz, ef - 994 - sf - lz, sg & 0x8000000000000000ull, odd);
                if (odd || ef >= dig::BAD_EXP) r = dig::special(r, ef);
                if (bad) r = __longlong_as_double(0x7FF8000000000000ll);
                if (dst[j]) {
                  *dst[j] = s[j] + r;
                  // the trace row of a boundary node is its face part
                  if (init && srow >= 0)
                    Se[((int64_t)dm.nu + (int64_t)sh.sblk[cb + j] * nb + srow) * ld + sh.scol[cb + j]] = r;
                }
              }
            }
          }
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&sh.dread);
        }
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 8) tc::tmem_dealloc(tmem, 256);
}

// Largest exponents of a pair's point coefficients: cu, cq_0, cq_1, cq_2 (3 Nq values each,
// contiguous), fuh, fq_0, fq_1, fq_2 and S_ik or lambda (Nfp each).  One warp per
// (element, pair).
__global__ void k_coef_exp(int Nq, int Nfp, AsmTab<double> tb, int16_t* __restrict__ out, int64_t n,
                           const int64_t* __restrict__ elist) {
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= n) return;
  int64_t e = w / 25;
  if (elist) {
    e = elist[e];
    if (e < 0) return;
  }
  const int64_t p = e * 25 + w % 25;
  for (int seg = 0; seg < 9; ++seg) {
    const double* src = seg < 4 ? tb.Jv + ((size_t)p * 12 + 3 * seg) * Nq
                                : (seg < 8 ? tb.Jf + ((size_t)p * 4 + (seg - 4)) * Nfp
                                           : (tb.Su ? tb.Su + (size_t)p * Nfp : tb.lamw + (size_t)e * Nfp));
    const int len = seg < 4 ? 3 * Nq : Nfp;
    const int* hi = reinterpret_cast<const int*>(src) + 1;
    int mx = 0;
    for (int i = lane; i < len; i += 32) mx = max(mx, hi[2 * i] & 0x7FF00000);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) out[p * 9 + seg] = (int16_t)(mx >> 20);
  }
}

// Largest exponents over the points of the lifted operators' columns (once per mesh).
__global__ void k_lift_exp(int Np, int Nb, int Nq, int Nfp, Geo G, int16_t* __restrict__ out, int64_t n) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n) return;
  const int w = Np + Nb, col = (int)(idx % w);
  const int64_t el = idx / w, e = el / 6;
  const int l = (int)(el % 3), pts = el % 6 < 3 ? Nq : Nfp, st = col < Np ? Np : Nb;
  const double* base = el % 6 < 3 ? (col < Np ? G.GlV : G.HlV) : (col < Np ? G.GlF : G.HlF);
  const double* src = base + ((size_t)e * 3 + l) * pts * st + (col < Np ? col : col - Np);
  int mx = 0;
  for (int g = 0; g < pts; ++g) mx = max(mx, dig::exponent_of(src[(size_t)g * st]));
  out[idx] = (int16_t)mx;
}

// x 2^(1023 - e) in FP32 from the upper word h of x, e >= 127: the lower mantissa bits are cut
// off (relative error 2^-20), values below FP32's range become 0.
__device__ __forceinline__ float norm32(int h, int e) {
  const int m = max((h & 0x7fffffff) - ((e - 127) << 20), 0);
  return __int_as_float((m << 3) | (h & (int)0x80000000));
}

// The exponents of the columns of V and W: em with |W| < 2^(em - 1022) for all points and
// directions, as low as possible (a bound from the factors' separate maxima was 6 bits too
// high on most columns and up to 15 on some, bits that the digits then lacked).  The sums
// are formed in FP32 in one scale per element: their error is below 2^-15 of the largest term
// a pair and column can have, and that, twice, is added to the largest one.  Pairs and columns
// too small for FP32 beside the element's others keep the bound from the maxima.
// A block takes an element, a warp 32 columns (lane = column) and a share of the points, with
// all pairs' maxima in registers; the coefficients go through shared memory 32 points at a
// time.  3D p = 3, 4096 elements 2.7 ms, p = 2, 2002 elements
// 0.5 ms, p = 4, 210 elements 0.5 ms (a warp per pair with the operators in shared memory: 6.4 ms
// at p = 3).
constexpr int WE_PTS = 32, WE_WARPS = 16;
template <int NP1, bool MIX>
__global__ void __launch_bounds__(32 * WE_WARPS, 2) k_w_exp(Dims dm, DgArgs a, int groups) {
  constexpr int NQ1 = NP1 + 1, Np = NP1 * NP1 * NP1, Nq = NQ1 * NQ1 * NQ1, Nfp = 6 * NQ1 * NQ1, m2 = 25;
  constexpr int NbU = Np - (NP1 - 2) * (NP1 - 2) * (NP1 - 2);
  __shared__ __align__(16) float sc[WE_PTS][m2][12];      // coefficients of a chunk of points
  extern __shared__ int smx[];                            // [25][columns] largest sums (bits of FP32)
  __shared__ int sref[3];                                 // largest exponents: basis value's coefficient, lifted, their coefficients
  const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int64_t slot = blockIdx.x, e = a.elist ? a.elist[slot] : slot;
  if (e < 0) return;
  const int NbT = MIX ? dm.Nb : NbU, nb = MIX ? a.tt.nb[e] : NbU, w = Np + NbT, ncol = Np + nb, C = 32 * groups;
  const int c = 32 * (warp % groups) + lane, share = warp / groups, shares = nth / C;
  const bool on = c < ncol, ucol = c < Np;
  const int col = ucol ? c : c - Np, bcol = ucol ? col : (MIX || !on ? 0 : a.ref.bnode[col]);
  const int gst = ucol ? Np : NbT;
  const int16_t* ec = a.ecoef + (size_t)e * m2 * 9;
  auto hi = [](const double* p) { return reinterpret_cast<const int*>(p)[1]; };
  auto has_cq = [](int pair) { return !(pair < 5 || (pair < 20 && pair % 5 == 4)); };
  auto points = [&](auto at_faces) {
    constexpr bool face = decltype(at_faces)::value;
    constexpr int n = face ? Nfp : Nq;
    const int16_t* eg = a.elift + ((size_t)e * 6 + 3 * face) * w;
    // the element's scale
    __syncthreads();
    if (tid < 3) sref[tid] = 0;
    for (int i = tid; i < m2 * C; i += nth) smx[i] = 0;
    __syncthreads();
    for (int i = tid; i < m2 * 9; i += nth) {
      const int seg = i % 9, x = ec[i];
      if (x != 0x7ff && (face ? seg >= 4 : seg < 4)) atomicMax(&sref[seg == 0 || seg == 4 || seg == 8 ? 0 : 2], x);
    }
    for (int i = tid; i < 3 * ncol; i += nth) atomicMax(&sref[1], (int)eg[(i / ncol) * w + i % ncol]);
    __syncthreads();
    const int scale = max(sref[0] + 1023, sref[2] + sref[1]);            // of a product, 2^(scale - 2046)
    const int e_bas = min(scale - 1023, 127 + 2047), e_lift = sref[1], e_coef = min(scale - e_lift, 127 + 2047);
    const bool fits = e_bas >= 127 && e_coef >= 127 && e_lift >= 127;
    const double* G = face ? (ucol ? a.tb.GlF + (size_t)e * 3 * Nfp * Np + col : a.tb.HlF + (size_t)e * 3 * Nfp * NbT + col)
                           : (ucol ? a.tb.GlV + (size_t)e * 3 * Nq * Np + col : a.tb.HlV + (size_t)e * 3 * Nq * NbT + col);
    const double* B = (face ? a.tb.PhiF : a.tb.Phi) + bcol;
    const bool basis = on && (face || ucol);
    float mx[m2];
#pragma unroll
    for (int p = 0; p < m2; ++p) mx[p] = 0.f;
    for (int g0 = 0; fits && g0 < n; g0 += WE_PTS) {
      const int cnt = min(WE_PTS, n - g0);
      __syncthreads();
      // volume: cu_0..2, cq_00 .. cq_22 (l slow); faces: fq_0..2, fuh, S_ik or lambda
      constexpr int per = face ? 5 : 12;
      for (int i = tid; i < per * m2 * WE_PTS; i += nth) {
        const int q = i % WE_PTS, k = (i / WE_PTS) % per, pair = i / (WE_PTS * per), g = g0 + q;
        if (q >= cnt) continue;
        const size_t ep = (size_t)e * m2 + pair;
        const double* src;
        if (!face) src = a.tb.Jv + (ep * 12 + k) * Nq + g;
        else if (k < 4) src = a.tb.Jf + (ep * 4 + (k + 1) % 4) * Nfp + g;
        else src = a.tb.Su ? a.tb.Su + ep * Nfp + g : a.tb.lamw + (size_t)e * Nfp + g;
        const bool none = face && k == 4 && a.tb.Su == nullptr && pair % 6 != 0;       // lambda delta_ik
        sc[q][pair][k] = none ? 0.f : norm32(hi(src), (face ? k >= 3 : k < 3) ? e_bas : e_coef);
      }
      __syncthreads();
      for (int q = share; q < cnt; q += shares) {
        const int g = g0 + q;
        float x[3];
#pragma unroll
        for (int l = 0; l < 3; ++l) {
          const float v = on ? norm32(hi(G + ((size_t)l * n + g) * gst), e_lift) : 0.f;
          x[l] = ucol ? -v : v;
        }
        const float b = basis ? norm32(hi(B + (size_t)g * Np), 1023) : 0.f;
#pragma unroll
        for (int p = 0; p < m2; ++p) {
          const float4 k0 = *reinterpret_cast<const float4*>(sc[q][p]);
          if constexpr (face) {
            float v = (ucol ? sc[q][p][4] : k0.w) * b;
            if (has_cq(p)) v = fmaf(k0.z, x[2], fmaf(k0.y, x[1], fmaf(k0.x, x[0], v)));
            mx[p] = fmaxf(mx[p], fabsf(v));
          } else {
            float v0 = k0.x * b, v1 = k0.y * b, v2 = k0.z * b;
            if (has_cq(p)) {
              const float4 k1 = *reinterpret_cast<const float4*>(sc[q][p] + 4), k2 = *reinterpret_cast<const float4*>(sc[q][p] + 8);
              v0 = fmaf(k2.y, x[2], fmaf(k1.z, x[1], fmaf(k0.w, x[0], v0)));
              v1 = fmaf(k2.z, x[2], fmaf(k1.w, x[1], fmaf(k1.x, x[0], v1)));
              v2 = fmaf(k2.w, x[2], fmaf(k2.x, x[1], fmaf(k1.y, x[0], v2)));
            }
            mx[p] = fmaxf(fmaxf(mx[p], fabsf(v0)), fmaxf(fabsf(v1), fabsf(v2)));
          }
        }
      }
    }
#pragma unroll
    for (int p = 0; p < m2; ++p) atomicMax(&smx[p * C + c], __float_as_int(mx[p]));
    __syncthreads();
    for (int i = tid; i < m2 * ncol; i += nth) {
      const int p = i / ncol, cc = i % ncol;
      const bool uc = cc < Np;
      // exponents of the pair's and column's terms; the largest real term is below 2^(top - 2044)
      const int eb = (face && uc) ? (a.tb.Su || p % 6 == 0 ? ec[p * 9 + 8] : 0) : (face || uc ? ec[p * 9 + (face ? 4 : 0)] : 0);
      int top = eb ? eb + 1023 : 0;
      bool bad = eb == 0x7ff;
      if (has_cq(p))
        for (int l = 0; l < 3; ++l) {
          const int el = ec[p * 9 + (face ? 5 : 1) + l], gl = eg[l * w + cc];
          if (el && gl) top = max(top, el + gl);
          bad |= el == 0x7ff;
        }
      int em = 0;
      if (top) {
        const int d = top - scale;
        em = top - 1019;
        if (fits && d > -90)
          em = min(em, scale - 1150 + (__float_as_int(__int_as_float(smx[p * C + cc]) + __int_as_float((127 + d - 14) << 23)) >> 23));
      }
      a.ew[(((size_t)slot * m2 + p) * 2 + (face ? 0 : 1)) * w + cc] = (int16_t)(bad ? 3 * 0x7ff : max(em, 0));
    }
  };
  if constexpr (!MIX) points(std::true_type{});
  points(std::false_type{});
}

template <int NP1>
cudaError_t dg_launch(iedg_mesh* M, const DgArgs& a, cudaStream_t st) {
  const Dims& dm = M->dm;
  const bool mix = M->tt.nb != nullptr;
  auto kern = mix ? k_assemble_dg<NP1, true> : k_assemble_dg<NP1, false>;
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DG_SMEM);
  if (err == cudaSuccess)
    err = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
  int dev = 0, sms = 0;
  if (err == cudaSuccess) err = cudaGetDevice(&dev);
  if (err == cudaSuccess) err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (err != cudaSuccess) return err;
  const int groups = idiv_up(dm.Np + dm.Nb, 32);       // of columns; as many warps as fit share the points
  if (groups > WE_WARPS) return cudaErrorInvalidValue;
  const size_t wsmem = sizeof(int) * 25 * 32 * (size_t)groups;
  auto wexp = mix ? k_w_exp<NP1, true> : k_w_exp<NP1, false>;
  err = cudaFuncSetAttribute(wexp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wsmem);
  if (err != cudaSuccess) return err;
  wexp<<<(unsigned)a.n_el, 32 * groups * (WE_WARPS / groups), wsmem, st>>>(dm, a, groups);
  err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  const int tiles = idiv_up(25 * (dm.Np + dm.Nb), DG_COLS);
  const int64_t n = a.n_el * tiles, g = 2 * (int64_t)sms;
  kern<<<(unsigned)(n < g ? n : g), DG_THREADS, DG_SMEM, st>>>(dm, a, tiles);
  return cudaGetLastError();
}

}  // namespace

bool assemble_dg_supported(const Dims& dm) { return dm.d == 3 && dm.p >= 2 && dm.p <= 4 && dm.nq1 == dm.p + 2; }

// Digits of the tables PhiF [Nfp][Np] and Dxi [3][Nq][Np] in operand order, their lanes'
// scales ([128] faces, [128] volume), and the number of volume chunks over which every
// level's sum stays below 2^24 whatever the other operand's digits are (the face chunks
// fit one window: a node's face values are zero on all but three faces).
void assemble_dg_table(const Dims& dm, const std::vector<double>& PhiF, const std::vector<double>& Dxi,
                       std::vector<unsigned char>& table, std::vector<int>& rexp, int* window) {
  const int Np = dm.Np, Nq = dm.Nq, Nfp = dm.Nfp, nfc = dg_face_chunks(Nfp), nvc = dg_vol_chunks(Nq);
  table.assign((size_t)(nfc + nvc) * 3 * DG_STEP_A, 0);
  rexp.assign(256, 0);
  auto bits = [](double x) { long long b; std::memcpy(&b, &x, 8); return b; };
  std::vector<double> mass((size_t)(nfc + nvc) * 128, 0.0);     // per chunk and lane: sum of |digits|
  auto put = [&](double x, int emax, int step, int a, int k) {
    const unsigned long long v = dig::to_bytes(bits(x), emax);
    for (int s = 0; s < dig::S; ++s) {
      const int d = (int)((v >> (8 * (7 - s))) & 0xff) - 128;
      const float f = (float)d;
      uint32_t u;
      std::memcpy(&u, &f, 4);
      const uint16_t b = (uint16_t)(u >> 16);
      std::memcpy(&table[(size_t)step * DG_STEP_A + s * DG_SLICE + dg_off(a, k)], &b, 2);
      mass[(size_t)(step / 3) * 128 + a] += std::abs(d);
    }
  };
  for (int a = 0; a < Np; ++a) {
    for (int fp = 0; fp < Nfp; ++fp) rexp[a] = std::max(rexp[a], dig::exponent_bits(bits(PhiF[(size_t)fp * Np + a])));
    for (size_t i = 0; i < (size_t)3 * Nq; ++i)
      rexp[128 + a] = std::max(rexp[128 + a], dig::exponent_bits(bits(Dxi[i * Np + a])));
    for (int fp = 0; fp < Nfp; ++fp) put(PhiF[(size_t)fp * Np + a], rexp[a], fp / DG_GP, a, fp % DG_GP);
    for (int r = 0; r < 3; ++r)
      for (int g = 0; g < Nq; ++g)
        put(Dxi[((size_t)r * Nq + g) * Np + a], rexp[128 + a], 3 * (nfc + g / DG_GP) + r, a, g % DG_GP);
  }
  for (*window = 4; *window > 1; *window /= 2) {
    double worst = 0.0;
    for (int c0 = 0; c0 < nvc; c0 += *window)
      for (int a = 0; a < 128; ++a) {
        double sum = 0.0;                // the last level meets every digit once
        for (int c = c0; c < std::min(nvc, c0 + *window); ++c) sum += mass[(size_t)(nfc + c) * 128 + a];
        worst = std::max(worst, 128.0 * sum);
      }
    if (worst <= 16777216.0) break;
  }
}

cudaError_t launch_lift_exp(iedg_mesh* M, cudaStream_t st) {
  const Dims& dm = M->dm;
  const int64_t n = M->E * 6 * (dm.Np + dm.Nb);
  k_lift_exp<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(dm.Np, dm.Nb, dm.Nq, dm.Nfp, M->geo, M->geo.elift, n);
  return cudaGetLastError();
}

// The element matrices of a uniform mesh, or the volume terms added to those of a mesh
// with mixed orders; elist != nullptr: of the listed elements, into their slots.
cudaError_t launch_assemble_dg(iedg_mesh* M, double* S, const int64_t* elist, int64_t n_slots, cudaStream_t st) {
  const Dims& dm = M->dm;
  const int64_t n_el = elist ? n_slots : M->E, nw = n_el * 25;
  const AsmTab<double> tb = tables64(M);
  k_coef_exp<<<(unsigned)((nw * 32 + 255) / 256), 256, 0, st>>>(dm.Nq, dm.Nfp, tb, M->pj.ecoef, nw, elist);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  const DgArgs a{tb, M->ref, M->pj.ecoef, M->geo.elift, M->pj.ew, elist ? M->rhs64 : nullptr, S, M->ph.alpha, M->tt, elist, n_el,
                 asm_wait_limit(M)};
  if (dm.p == 2) return dg_launch<3>(M, a, st);
  if (dm.p == 3) return dg_launch<4>(M, a, st);
  return dg_launch<5>(M, a, st);
}

}  // namespace iedg
