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
//   * a column's scale is a bound on its largest |W| from the exponents of its factors
//     (largest exponents per pair, and per column of Gl, Hl), so W is converted as it is
//     formed; the bound costs a few of the 62 digit bits;
//   * FP32 level sums stay exact (below 2^24) over a window of chunks, checked for the
//     tables' own digits when they are laid out; then the levels are joined in 96-bit
//     integers, rounded once to FP64 and added to the element matrix.
// Warps: 8 form and convert W and read the accumulators, one issues the MMAs, one the
// copies; they meet at mbarriers, all waits bounded.  Two CTAs per SM, so that one's
// conversion and results overlap the other's FP64.
// Meshes with mixed orders have trace bases of their own: there the face terms come from
// k_assemble_sf first and this kernel adds the volume terms.
// Measured, all elements, sum-factorised on the FP64 pipe -> this kernel: 3D p = 3, 4096
// elements 135.4 -> 95.8 ms; p = 2, 2002 elements 14.0 -> 12.4 ms; p = 4, 210 elements 32.8 ->
// 17.2 ms; orders 2, 3, 4 mixed, 324 elements 25.6 -> 16.8 ms.  Counters at p = 3: FP64 pipe
// 50 % busy, tensor pipe 26 %, 7.9 TB/s from L2, two thirds of it the tables.
#include <algorithm>
#include <cstdlib>
#include <cstring>

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
    if (!tc::mbar_wait(bar, parity & 1u, *failed ? 1 : a.wait_limit)) *failed = 1;
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
          if (q >= DG_RING) wait(&sh.empty[st], q / DG_RING - 1);
          if (*failed) break;
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
          if (start && nwin > 0) wait(&sh.dread, nwin - 1);   // accumulators read
          wait(&sh.bfull, nch);                               // W of this chunk staged
          const bool end = window_end(ch, ch1);
          for (int r = 0; r < 3 && !*failed; ++r, ++q) {
            const uint32_t st = q % DG_RING;
            wait(&sh.full[st], q / DG_RING);
            if (*failed) break;
            tc::fence_after_sync();
#pragma unroll
            for (int s = 0; s < dig::S; ++s)
              tc::mma_bf16(tmem + (uint32_t)(s * DG_COLS), da0 + (uint64_t)((st * DG_STEP_A + s * DG_SLICE) >> 4),
                           db0 + (uint64_t)((r * DG_STEP_B) >> 4), tc::idesc_bf16(128, DG_COLS * (dig::S - s)),
                           (start && r == 0 && s == 0) ? 0u : 1u);
            tc::mma_commit(&sh.empty[st]);
          }
          if (*failed) break;
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
      // scales: |W| <= 4 max of the terms; a term's exponent is at most ea + eb + 1, that of
      // a basis value (below 2) 1023; one more for the terms' rounding
      int emV = 0, emF = 0;
      if (on) {
        const int16_t* ec = a.ecoef + ep * 9;
        const int16_t* eg = a.elift + (size_t)e * 6 * (Np + NbT) + (ucol ? col : Np + col);
        auto term = [](int ea, int eb) { return ea == 0x7ff ? 3 * 0x7ff : ea + eb - 1022; };
        if (ucol) emV = term(ec[0], 1023);
        if (fu) emF = term(ec[ucol ? 8 : 4], 1023);
        if (cq)
#pragma unroll
          for (int l = 0; l < 3; ++l) {
            emV = max(emV, term(ec[1 + l], eg[l * (Np + NbT)]));
            emF = max(emF, term(ec[5 + l], eg[(3 + l) * (Np + NbT)]));
          }
        emV += 3;
        emF += 3;
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
        if (nch > 0) wait(&sh.bempty, nch - 1);                 // the MMAs have read the previous chunk
        const int em = face ? emF : emV;
        if (!*failed) {
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            const unsigned long long v0 = dig::to_bytes(__double_as_longlong(w[r][0]), em);
            const unsigned long long v1 = dig::to_bytes(__double_as_longlong(w[r][1]), em);
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
          wait(&sh.dfull, nwin++);
          tc::fence_after_sync();
          if (32 * qt < Np) {
            const bool bad = *failed != 0;
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
  const DgArgs a{tb, M->ref, M->pj.ecoef, M->geo.elift, elist ? M->rhs64 : nullptr, S, M->ph.alpha, M->tt, elist, n_el,
                 asm_wait_limit(M)};
  if (dm.p == 2) return dg_launch<3>(M, a, st);
  if (dm.p == 3) return dg_launch<4>(M, a, st);
  return dg_launch<5>(M, a, st);
}

}  // namespace iedg
