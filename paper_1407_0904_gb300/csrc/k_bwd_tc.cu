// FP64 adjoint on the tensor cores: Gbar_e[k] = sum_o T[k][o] dA_e[o] by exact digit products (the method of
// k_fp64_tc.cu), then the chain rule to vertices and coefficients in FP64.
//
// The plain FP64 kernel (k_bwd.cu) is bound by the FP64 pipe, 2 FMAs per cycle and SM: advection-diffusion
// P2 on tetrahedra takes K N = 3600 of them per cell for Gbar and about 370 for the chain, 1.41 ms for 196,608
// cells whose dA is read in 23 us. Here the contraction runs on the tensor cores over digits of dA (62-bit
// fixed point, eight 8-bit digits), and the chain is rewritten on the adjugate A and the determinant
// (K = A / det), about 280 operations: 0.206 ms. FP64 remains the bound there, now for the chain alone (0.11
// ms) and for what does not overlap it; Helmholtz P2 (0.326 -> 0.128 ms) is bound by the making of the digits
// and the scan.
//
// Tiles of 128 cells on the TMEM lanes (M = 128), the factors k on the columns (16 or 48): per order d = p + q < 8
// one accumulator of K columns. Entries o come in parts of 16, each a stage of the cells' digits and of T's
// (copied in bulk from its image); seven parts (112 entries) is what an FP32 accumulator sums exactly
// (112 * 8 * 2^14 < 2^24), so each cell's exponent is that of 112 entries, after which the orders are drained,
// combined in 64-bit integers and rounded to double (with more than 112 entries the drains are added in FP64,
// one rounding per 112 entries where the plain kernel rounds every one). Errors against 64-bit autograd are the
// plain kernel's or smaller (1.0e-15 and 1.1e-15 for advection-diffusion P2).
// An error relative to the largest dA of a row is a rounding of Gbar[k]'s own terms only if some large dA meets a large
// T[k]. The scan looks for one for every k; cells without (one entry far above the others, a single row of dA) take
// the plain sums, alone by the scan's warp (whole_cell), many by a lane each (plain_gbar: with one row of dA alone
// in every cell 0.3-1.1 times the plain kernel's time on tetrahedra, with six decades of spread 1.2-1.5). The check costs up to a quarter: us for 196,608 tetrahedra without / with it, advection-
// diffusion P1 164 / 221, P2 193 / 206, P3 584 / 670, Helmholtz P1 88 / 104, P2 124 / 128.
//   warps 0-7    epilogue, two sets on alternate tiles (one drains while the other is in the FP64 chain);
//                a thread has one cell: drains, chain rule, atomics or local rows
//   warps 8-11   producers: digits of dA (this second reading of it hits L2)
//   warps 12-14  scan: the largest exponent of each cell's dA, the k with a large dA at a large T[k]
//   warp 15      MMA issue
#include <cuda_runtime.h>
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include "coffee_internal.h"
#include "tc_common.cuh"
#include "fp64_common.cuh"
#include "digits.cuh"

namespace coffee {
namespace {

using namespace tc;

constexpr int G_ND = 8, G_FB = 62;  // 8-bit digits, fraction bits
constexpr int G_PE = 16;             // entries per part
constexpr int G_CH = G_PE / 4;       // 16-byte chunks per part and digit pair: 4 entries x 2 digits
constexpr int G_DRAIN = 7;           // parts between drains
constexpr int G_STAGES = 4;         // at most
constexpr int G_EPI = 8, G_PROD = 4, G_SCAN = 3;
constexpr int G_WARPS = G_EPI + G_PROD + G_SCAN + 1;  // 16: four per scheduler, 128 registers a thread
constexpr int G_THREADS = G_WARPS * 32;
constexpr int G_XRING = 4;           // drains whose cell exponents are kept
constexpr int G_SH = 43;             // weight of order 0 in a drain's 64-bit sum (112 * 65^2 * 2^43 < 2^62)
constexpr int G_ASTAGE = G_ND / 2 * G_CH * BM * 16;
constexpr uint64_t G_BIAS = 0x8080808080808080ull;
constexpr int CELL_PLAIN = INT32_MIN, CELL_DONE = INT32_MIN + 1;  // instead of an exponent: for plain_gbar; by the scan (whole_cell)
constexpr int G_WEAK_A = 4, G_WEAK_T = 2;  // dA counts as large above 2^-4 of its drain's largest, T[k] above 2^-2 of its own

struct alignas(8) GBars {
  uint64_t full[G_STAGES], empty[G_STAGES], tfull[2][2], tempty[2], xfull[G_XRING], xempty[G_XRING], done;  // tfull[set of warps][buffer]
  uint32_t tmem_base;
};

template <int FORM, int D>
struct Adj {
  static constexpr int K = FormK<FORM, D>::value, NV = D + 1;
  static constexpr int NC = (K + 15) / 16 * 16;             // accumulator columns of one order
  static constexpr int BUFS = 2 * G_ND * NC <= 512 ? 2 : 1;  // tiles in TMEM at a time
  static constexpr int TSTAGE = G_CH * G_ND * NC * 16;      // bytes of one part of T's image
  static constexpr int STAGE = G_ASTAGE + TSTAGE;
  static constexpr int STAGES = G_STAGES * STAGE <= 200 * 1024 ? G_STAGES : 3;
  static constexpr int NCF = FORM == FORM_ADVDIFF ? NV * (1 + D) : 0;
  static constexpr int NL = NV * D + NCF;
  static constexpr int KP = (K + 1) / 2 * 2;                // words of an entry's row in the transposed T
};

// expects bytes in the barrier's current phase, without arriving (this thread's arrival follows its own stores)
__device__ __forceinline__ void g_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void g_bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// Entries o and o + 1 of a row of N (o even), zero past its end. vec: rows start on 16 bytes.
__device__ __forceinline__ void load_pair(const double* row, int o, int N, bool vec, double& a, double& b) {
  if (vec) {
    const double2 w = o < N ? __ldg(reinterpret_cast<const double2*>(row + o)) : make_double2(0.0, 0.0);
    a = w.x;
    b = w.y;
  } else {
    a = o < N ? __ldg(row + o) : 0.0;
    b = o + 1 < N ? __ldg(row + o + 1) : 0.0;
  }
}

// x as a fixed-point number of 62 fraction bits below the cell's largest exponent X (in place), plus the
// digits' bias; an exponent far below X, subnormals among them, shifts x out.
__device__ __forceinline__ uint64_t fixed62(double x, int X) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const uint32_t sh = ((uint32_t)X - (h & 0x7FF00000u)) >> 20, s = (uint32_t)((int)h >> 31);
  uint64_t m = (uint64_t)((h & 0xFFFFFu) | 0x100000u) << 32 | l;
  asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m << 9), "r"(sh));  // (clamps)
  return (m ^ ((uint64_t)s << 32 | s)) + G_BIAS;                // -m less one in the last place for negative x
}

// Two numbers' digits in pairs (0,1), (2,3), (4,5), (6,7): a word for each number and pair with the pair's
// leading digit in its low half, in the pair's chunk. A digit is a byte u of the biased number; a byte
// permutation puts two of them below 0x64, which makes the halves 1024 + u, and one packed subtraction leaves
// u - 128.
__device__ __forceinline__ void store_pairs(uint8_t* dst, uint64_t U0, uint64_t U1) {
  const __half2 off = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));
#pragma unroll
  for (int P = 0; P < 4; ++P) {
    uint32_t w[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint64_t U = j ? U1 : U0;
      const uint32_t u = __byte_perm(P < 2 ? (uint32_t)(U >> 32) : (uint32_t)U, 0x64646464u, P & 1 ? 0x4041u : 0x4243u);
      const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&u), off);
      w[j] = *reinterpret_cast<const uint32_t*>(&v);
    }
    *reinterpret_cast<uint2*>(dst + P * G_CH * BM * 16) = make_uint2(w[0], w[1]);
  }
}

// Bit of entry o of a drain in the masks of large entries: 16 bits for each of the eight lanes that scan a row
COFFEE_HD inline int mask_bit(int o, bool vec) { return vec ? o % 16 / 2 * 16 + o / 16 * 2 + o % 2 : o % 8 * 16 + o / 8; }

// Gbar of a cell whose dA the digits do not take: not finite, outside 2^+-900, or without a large entry where some T[k] is
// large. T's rows by entry: by factor, one such cell of P3 tetrahedra (N = 400) alone took 800,000 cycles, 36 lines an entry.
template <int FORM, int D>
__device__ __noinline__ void plain_gbar(const BwdParams& p, int64_t e, double* Gb) {
  constexpr int K = Adj<FORM, D>::K, KP = Adj<FORM, D>::KP;
  const double* row = static_cast<const double*>(p.dout) + e * p.N;
  const double2* T = static_cast<const double2*>(p.rows);
  double s[KP];
#pragma unroll
  for (int k = 0; k < KP; ++k) s[k] = 0.0;
  constexpr int U = K <= 16 ? 4 : 1;  // entries whose loads are issued together
  for (int o = 0; o < p.N; o += U) {
    double a[U];
    bool some = false;
#pragma unroll
    for (int j = 0; j < U; ++j) {
      a[j] = o + j < p.N ? __ldg(row + o + j) : 0.0;
      some = some || a[j] != 0.0;
    }
    if (!some) continue;  // (dA of a few rows or columns is what comes here most)
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int r = U == 1 || o + j < p.N ? o + j : o;  // past the end: any row, by zero
#pragma unroll
      for (int k = 0; k < KP; k += 2) {
        const double2 t = __ldg(T + r * (KP / 2) + k / 2);
        s[k] = fma(t.x, a[j], s[k]);
        s[k + 1] = fma(t.y, a[j], s[k + 1]);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) Gb[k] = s[k];
}

// Chain rule of one cell, from Gbar to the local gradient L (vertex coordinates v*D + r, then eps_v, then
// b_{v,r}). With J, its adjugate A and det, s = sign(det), per cell
//   G_mass = |det|, H_ab = (A A^T)_ab / |det|, G_stiff = eps_v H_ab, G_adv[v,a] = s sum_r A[a][r] b_v[r]:
//   S = the symmetric matrix of sum_v eps_v Gbar_stiff (off-diagonals halved),
//   W = dL/dA = 2/|det| S A + s sum_v Gbar_adv[v] b_v^T,   dL/d|det| = Gbar_mass - <S, H>/|det|,
//   dL/dJ = the cofactors' derivative applied to W, plus s dL/d|det| A^T.
template <int FORM, int D>
__device__ __forceinline__ void chain_rule(const double (&X)[D + 1][D], const BwdParams& p, const int (&cid)[D + 1],
                                           const double (&Gb)[FormK<FORM, D>::value], double (&L)[Adj<FORM, D>::NL]) {
  constexpr int NV = D + 1, P = D * (D + 1) / 2;
  double J[D][D], W[D][D];
#pragma unroll
  for (int r = 0; r < D; ++r)
#pragma unroll
    for (int c = 0; c < D; ++c) J[r][c] = X[c + 1][r] - X[0][r];
  Geo<D> g;
  geometry64<D>(X, g);
  const double Dm = fabs(g.det), s = g.det < 0.0 ? -1.0 : 1.0, inv = 1.0 / Dm;
  double db = FORM == FORM_ADVDIFF ? 0.0 : Gb[0];  // dL/d|det|
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int r = 0; r < D; ++r) W[a][r] = 0.0;
  if constexpr (FORM != FORM_MASS) {
    double S[P], H[P];
#pragma unroll
    for (int q = 0; q < P; ++q) {
      if constexpr (FORM == FORM_HELMHOLTZ) {
        S[q] = Gb[1 + q];
      } else {
        S[q] = 0.0;
#pragma unroll
        for (int v = 0; v < NV; ++v) S[q] = fma(__ldg(p.coef + (int64_t)cid[v] * (D + 1)), Gb[v * P + q], S[q]);
      }
    }
    double t = 0.0;
    int q = 0;
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
      for (int b = a; b < D; ++b, ++q) {
        double h = 0.0;
#pragma unroll
        for (int r = 0; r < D; ++r) h = fma(g.adj[a][r], g.adj[b][r], h);
        H[q] = h * inv;
        t = fma(S[q], H[q], t);
        const double c = S[q] * inv;  // 2/|det| S A: the halved off-diagonals count twice
#pragma unroll
        for (int r = 0; r < D; ++r) {
          W[a][r] = fma(c, a == b ? 2.0 * g.adj[b][r] : g.adj[b][r], W[a][r]);
          if (a != b) W[b][r] = fma(c, g.adj[a][r], W[b][r]);
        }
      }
    db = fma(-t, inv, db);
    if constexpr (FORM == FORM_ADVDIFF) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        double e = 0.0;
#pragma unroll
        for (int k = 0; k < P; ++k) e = fma(Gb[v * P + k], H[k], e);
        L[NV * D + v] = e;
        double ga[D];
#pragma unroll
        for (int a = 0; a < D; ++a) ga[a] = s * Gb[NV * P + v * D + a];
#pragma unroll
        for (int r = 0; r < D; ++r) {
          const double b = __ldg(p.coef + (int64_t)cid[v] * (D + 1) + 1 + r);
          double x = 0.0;
#pragma unroll
          for (int a = 0; a < D; ++a) {
            W[a][r] = fma(ga[a], b, W[a][r]);
            x = fma(ga[a], g.adj[a][r], x);
          }
          L[NV * D + NV + v * D + r] = x;
        }
      }
    }
  }
  double Jb[D][D];
  const double sd = s * db;
#pragma unroll
  for (int r = 0; r < D; ++r)
#pragma unroll
    for (int c = 0; c < D; ++c) Jb[r][c] = sd * g.adj[c][r];
  if constexpr (FORM != FORM_MASS) {
    if constexpr (D == 2) {
      Jb[1][1] += W[0][0];
      Jb[0][1] -= W[0][1];
      Jb[1][0] -= W[1][0];
      Jb[0][0] += W[1][1];
    } else {
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int r = 0; r < 3; ++r) {  // A[a][r] = J[r1][a1] J[r2][a2] - J[r1][a2] J[r2][a1]
          const int r1 = (r + 1) % 3, r2 = (r + 2) % 3, a1 = (a + 1) % 3, a2 = (a + 2) % 3;
          Jb[r1][a1] = fma(W[a][r], J[r2][a2], Jb[r1][a1]);
          Jb[r2][a2] = fma(W[a][r], J[r1][a1], Jb[r2][a2]);
          Jb[r1][a2] = fma(-W[a][r], J[r2][a1], Jb[r1][a2]);
          Jb[r2][a1] = fma(-W[a][r], J[r1][a2], Jb[r2][a1]);
        }
    }
  }
#pragma unroll
  for (int r = 0; r < D; ++r) {
    double x = 0.0;
#pragma unroll
    for (int c = 0; c < D; ++c) {
      L[(c + 1) * D + r] = Jb[r][c];
      x += Jb[r][c];
    }
    L[r] = -x;
  }
}

// The local gradient from Gbar, to the cell's local row or added to the vertices' and coefficients' gradients
template <int FORM, int D>
__device__ __forceinline__ void finish_cell(const BwdParams& p, int64_t e, const int (&vid)[D + 1], const int (&cid)[D + 1],
                                            const double (&X)[D + 1][D], const double (&Gb)[FormK<FORM, D>::value]) {
  constexpr int NV = D + 1, NL = Adj<FORM, D>::NL;
  double L[NL];
  chain_rule<FORM, D>(X, p, cid, Gb, L);
  if (p.local) {  // deterministic mode: summed later in cell order
#pragma unroll
    for (int j = 0; j < NL; ++j) p.local[e * NL + j] = L[j];
  } else {
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int r = 0; r < D; ++r) atomicAdd(p.d_coords + (int64_t)vid[v] * D + r, L[v * D + r]);
    if constexpr (FORM == FORM_ADVDIFF) {
      if (p.d_coef) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          double* dc = p.d_coef + (int64_t)cid[v] * (D + 1);
          atomicAdd(dc, L[NV * D + v]);
#pragma unroll
          for (int r = 0; r < D; ++r) atomicAdd(dc + 1 + r, L[NV * D + NV + v * D + r]);
        }
      }
    }
  }
}

// One cell without digits by a whole warp. Alone in a warp of the epilogue it would hold up a tile (plain_gbar takes 700,000
// cycles of latency for N = 400: with one cell in 10,000, advection-diffusion P3 on 196,608 tetrahedra took 1290 us,
// now 670).
template <int FORM, int D>
__device__ __noinline__ void whole_cell(const BwdParams& p, int64_t e) {
  constexpr int K = Adj<FORM, D>::K, NV = D + 1;
  const double* row = static_cast<const double*>(p.dout) + e * p.N;
  double Gb[K];
#pragma unroll
  for (int k = 0; k < K; ++k) Gb[k] = 0.0;
  for (int o = threadIdx.x & 31; o < p.N; o += 32) {
    const double a = __ldg(row + o);
#pragma unroll
    for (int k = 0; k < K; ++k) Gb[k] = fma(__ldg(p.T + (int64_t)k * p.N + o), a, Gb[k]);
  }
  __syncwarp();
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int m = 16; m > 0; m /= 2) Gb[k] += __shfl_xor_sync(0xffffffffu, Gb[k], m);
  if ((threadIdx.x & 31) == 0) {
    int vid[NV], cid[NV];
    bool bad = false;  // (which the epilogue reports)
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      vid[v] = __ldg(p.c2v + e * NV + v);
      cid[v] = FORM == FORM_ADVDIFF ? __ldg(p.c2d + e * NV + v) : 0;
      if (p.validate && (vid[v] < 0 || vid[v] >= p.nverts || (FORM == FORM_ADVDIFF && (cid[v] < 0 || cid[v] >= p.ncoefnodes)))) bad = true;
    }
    if (!bad) {
      double X[NV][D];
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int r = 0; r < D; ++r) X[v][r] = __ldg(p.coords + (int64_t)vid[v] * D + r);
      finish_cell<FORM, D>(p, e, vid, cid, X, Gb);
    }
  }
  __syncwarp();
}

template <int FORM, int D>
__global__ void __launch_bounds__(G_THREADS, 1) k_backward_tc(const BwdParams p) {
  using AF = Adj<FORM, D>;
  constexpr int K = AF::K, NC = AF::NC, NV = AF::NV, NL = AF::NL, BUFS = AF::BUFS;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* sS = smem_raw;
  int* sX = reinterpret_cast<int*>(sS + AF::STAGES * AF::STAGE);
  uint4* sT = reinterpret_cast<uint4*>(sX + G_XRING * BM);            // masks of T's large entries [drain][k]
  const int ndr = ((p.N + G_PE - 1) / G_PE + G_DRAIN - 1) / G_DRAIN;
  uint4* sL = sT + ndr * K;                                           // of dA's, of the eight rows a scan warp is at
  int4* sR = reinterpret_cast<int4*>(sL + G_SCAN * 8);                // a row's scale and factors so far [BM]
  GBars* bars = reinterpret_cast<GBars*>(sR + BM);

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int N = p.N;
  const int nparts = (N + G_PE - 1) / G_PE, ndrains = ndr;
  const bool vec = (N & 1) == 0 && (reinterpret_cast<uintptr_t>(p.dout) & 15) == 0;  // rows that can be read in pairs
  const int64_t ntiles = (p.ncells + BM - 1) / BM;

  {
    const uint4* src = reinterpret_cast<const uint4*>(p.large) + (vec ? 0 : ndrains * K);
    for (int i = threadIdx.x; i < ndrains * K; i += G_THREADS) sT[i] = __ldg(src + i);
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < G_STAGES; ++s) {
      mbar_init(smem_u32(&bars->full[s]), BM);
      mbar_init(smem_u32(&bars->empty[s]), 1);
    }
    for (int r = 0; r < 2; ++r) {
      mbar_init(smem_u32(&bars->tfull[0][r]), 1);
      mbar_init(smem_u32(&bars->tfull[1][r]), 1);
      mbar_init(smem_u32(&bars->tempty[r]), 4);
    }
    for (int r = 0; r < G_XRING; ++r) {
      mbar_init(smem_u32(&bars->xfull[r]), G_SCAN);
      mbar_init(smem_u32(&bars->xempty[r]), 4);
    }
    mbar_init(smem_u32(&bars->done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == G_WARPS - 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tmem_base)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  const uint32_t full = smem_u32(bars->full), empty = smem_u32(bars->empty);
  const uint32_t tfull = smem_u32(bars->tfull), tempty = smem_u32(bars->tempty);
  const uint32_t xfull = smem_u32(bars->xfull), xempty = smem_u32(bars->xempty);

  if (warp >= G_EPI && warp < G_EPI + G_PROD) {
    // ---------------- producers: 32 cells per warp, four lanes and two entries a lane per cell ----------------
    // (a lane per cell reads as many bytes, but every load then touches 32 lines: L1 took 1000 cycles a part)
    // (half warps store 128 contiguous bytes: rows 0-7, the chunk of pr 0 and 1 or of pr 2 and 3)
    const int w = warp - G_EPI, r8 = (lane >> 1) & 7, pr = (lane & 1) | (lane >> 4) << 1;
    uint32_t n = 0, dr = 0;  // parts stored, drains begun
    bool ok = true;
    for (int64_t t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      const int64_t e0 = t * BM + w * 32 + r8;  // this lane's cells: e0, e0 + 8, e0 + 16, e0 + 24
      const double* src = static_cast<const double*>(p.dout) + e0 * N;
      double v[4][4];  // [cell][entries 2 pr, 2 pr + 1 of the part's first and second eight]
      auto load_part = [&](int part) {
        const int o = part * G_PE + 2 * pr;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int cols = e0 + 8 * c < p.ncells ? N : 0;
#pragma unroll
          for (int h = 0; h < 2; ++h) load_pair(src + (int64_t)(8 * c) * N, o + 8 * h, cols, vec, v[c][2 * h], v[c][2 * h + 1]);
        }
      };
      load_part(0);
      int X[4];
      for (int part = 0; part < nparts; ++part, ++n) {
        if (part % G_DRAIN == 0) {
          const int r = (int)(dr % G_XRING);
          if (!mbar_wait(xfull + 8 * r, (dr / G_XRING) & 1u, p.err)) { ok = false; break; }
          ++dr;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            // rows without digits (zero, or left to plain_gbar) take an exponent that shifts everything out
            const int x20 = sX[r * BM + w * 32 + 8 * c + r8];
            X[c] = x20 > -(1022 << 20) ? x20 + (1022 << 20) : 0x7FE00000;
          }
        }
        const int st = n % AF::STAGES;
        uint64_t U[4][4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int j = 0; j < 4; ++j) U[c][j] = fixed62(v[c][j], X[c]);
        load_part(part + 1);  // requested before this part is stored
        if (!mbar_wait(empty + 8 * st, ((n / AF::STAGES) & 1u) ^ 1u, p.err)) { ok = false; break; }
        uint8_t* stage = sS + st * AF::STAGE;
        if (w == 0 && lane == 0) {
          g_expect_tx(full + 8 * st, AF::TSTAGE);
          g_bulk_g2s(smem_u32(stage + G_ASTAGE), p.digits + (size_t)part * AF::TSTAGE, AF::TSTAGE, full + 8 * st);
        }
        uint8_t* dst = stage + (pr >> 1) * (BM * 16) + (w * 32 + r8) * 16 + (pr & 1) * 8;
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int h = 0; h < 2; ++h) store_pairs(dst + 2 * h * (BM * 16) + 8 * c * 16, U[c][2 * h], U[c][2 * h + 1]);
        fence_proxy_async();
        mbar_arrive(full + 8 * st);
      }
    }
    // no copy may land after this block has left (its waits may have expired): wait for the last one of each stage
    if (w == 0 && lane == 0)
      for (uint32_t k = n > (uint32_t)AF::STAGES ? n - AF::STAGES : 0; k < n; ++k)
        mbar_wait(full + 8 * (k % AF::STAGES), (k / AF::STAGES) & 1u, p.err);
    __syncwarp();
  } else if (warp >= G_EPI + G_PROD && warp < G_WARPS - 1) {
    // ---------------- scan: the largest exponent of every cell's dA in a drain's entries, drains ahead ----------------
    // A drain's error is 2^-55 of max|T[k]| times its own largest |dA|: no more than roundings of sum_o |T[k][o] dA[o]| where a
    // drain of at least half that scale has a large dA at a large T[k]. So the scan also finds, per row and drain, the k for
    // which one has (a lane per k, masks of 112 entries), and leaves cells with a k for which none has to plain_gbar.
    const int w = warp - (G_EPI + G_PROD);
    const double* dA = static_cast<const double*>(p.dout);
    uint32_t dr = 0;
    bool ok = true;
    for (int64_t t = blockIdx.x; t < ntiles && ok; t += gridDim.x)
    for (int dn = 0; dn < ndrains; ++dn, ++dr) {
      const int r = (int)(dr % G_XRING), o1 = dn * (G_DRAIN * G_PE), len = min(N - o1, G_DRAIN * G_PE);
      ok = __all_sync(0xffffffffu, mbar_wait(xempty + 8 * r, ((dr / G_XRING) & 1u) ^ 1u, p.err));
      if (!ok) break;
      const uint4 none = make_uint4(0, 0, 0, 0);
      const uint4 t0 = lane < K ? sT[dn * K + lane] : none, t1 = lane + 32 < K ? sT[dn * K + lane + 32] : none;
      // Eight rows at a time, eight lanes each on two of them, and 16 predicated loads in flight: the scan is
      // bound by their latency (one row a time and a loop left to the compiler, which takes short rows one
      // load at a time, took 34,000 cycles a tile of 100 entries, half the kernel's time).
      for (int row0 = 8 * w; row0 < BM; row0 += 8 * G_SCAN) {
        const int row = row0 + (lane >> 3);
        const int64_t e = t * BM + row;
        const double* src = dA + e * N + o1;
        const int colsA = e < p.ncells ? len : 0, colsB = e + 4 < p.ncells ? len : 0;
        const double* srcB = src + (int64_t)4 * N;
        int X[2] = {0, 0}, some[2] = {0, 0};  // largest magnitude's high word; low words
        {
          // the next drain's lines of these rows on their way to L2: scanned from DRAM, eight rows took 3700
          // cycles of latency, 22,000 a drain, more than any other role
          const int64_t en = dn + 1 < ndrains ? e : e + (int64_t)gridDim.x * BM;
          const int on = dn + 1 < ndrains ? o1 + G_DRAIN * G_PE : 0, at = on + 16 * (lane & 7);
          if (at < min(N, on + G_DRAIN * G_PE)) {
            const double* nx = dA + en * N + at;
            if (en < p.ncells) asm volatile("prefetch.global.L2 [%0];" ::"l"(nx));
            if (en + 4 < p.ncells) asm volatile("prefetch.global.L2 [%0];" ::"l"(nx + (int64_t)4 * N));
          }
        }
        auto over_row = [&]() {
#pragma unroll
          for (int m = 1; m < 8; m *= 2)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              X[j] = max(X[j], __shfl_xor_sync(0xffffffffu, X[j], m));
              some[j] |= __shfl_xor_sync(0xffffffffu, some[j], m);
            }
        };
        uint32_t large[2] = {0, 0};  // this lane's entries above 2^-4 of the row's largest
        if (vec) {
          const int o0 = 2 * (lane & 7);
          int4 b[2][7];
#pragma unroll
          for (int j = 0; j < 7; ++j) {
            b[0][j] = o0 + 16 * j < colsA ? __ldg(reinterpret_cast<const int4*>(src + o0 + 16 * j)) : make_int4(0, 0, 0, 0);
            b[1][j] = o0 + 16 * j < colsB ? __ldg(reinterpret_cast<const int4*>(srcB + o0 + 16 * j)) : make_int4(0, 0, 0, 0);
          }
#pragma unroll
          for (int j = 0; j < 14; ++j) {
            const int4 c = b[j & 1][j >> 1];
            X[j & 1] = max(X[j & 1], max(c.y & 0x7FFFFFFF, c.w & 0x7FFFFFFF));
            some[j & 1] |= c.x | c.z;
          }
          over_row();
#pragma unroll
          for (int j = 0; j < 14; ++j) {
            const int4 c = b[j & 1][j >> 1];
            const int least = X[j & 1] - (G_WEAK_A << 20);
            large[j & 1] |= ((c.y & 0x7FFFFFFF) >= least ? 1u << (j & ~1) : 0u) | ((c.w & 0x7FFFFFFF) >= least ? 2u << (j & ~1) : 0u);
          }
        } else {
          const int o0 = lane & 7;
          int2 b[2][14];
#pragma unroll
          for (int j = 0; j < 14; ++j) {
            b[0][j] = o0 + 8 * j < colsA ? __ldg(reinterpret_cast<const int2*>(src + o0 + 8 * j)) : make_int2(0, 0);
            b[1][j] = o0 + 8 * j < colsB ? __ldg(reinterpret_cast<const int2*>(srcB + o0 + 8 * j)) : make_int2(0, 0);
          }
#pragma unroll
          for (int j = 0; j < 28; ++j) {
            const int2 c = b[j & 1][j >> 1];
            X[j & 1] = max(X[j & 1], c.y & 0x7FFFFFFF);
            some[j & 1] |= c.x;
          }
          over_row();
#pragma unroll
          for (int j = 0; j < 28; ++j)
            large[j & 1] |= (b[j & 1][j >> 1].y & 0x7FFFFFFF) >= X[j & 1] - (G_WEAK_A << 20) ? 1u << (j >> 1) : 0u;
        }
        uint16_t* masks = reinterpret_cast<uint16_t*>(sL + w * 8);
#pragma unroll
        for (int j = 0; j < 2; ++j) masks[((lane >> 3) + 4 * j) * 8 + (lane & 7)] = (uint16_t)large[j];
        __syncwarp();
        uint32_t lo = 0, hi = 0;  // of row row0 + lane, lanes 0 to 7: the k with a large dA at a large T[k]
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint4 m = sL[w * 8 + j];
          const uint32_t g0 = __ballot_sync(0xffffffffu, ((t0.x & m.x) | (t0.y & m.y) | (t0.z & m.z) | (t0.w & m.w)) != 0u);
          if (lane == j) lo = g0;
          if constexpr (K > 32) {
            const uint32_t g1 = __ballot_sync(0xffffffffu, ((t1.x & m.x) | (t1.y & m.y) | (t1.z & m.z) | (t1.w & m.w)) != 0u);
            if (lane == j) hi = g1;
          }
        }
        const int xa = __shfl_sync(0xffffffffu, X[0], (lane & 3) * 8), xb = __shfl_sync(0xffffffffu, X[1], (lane & 3) * 8);
        const int sa = __shfl_sync(0xffffffffu, some[0], (lane & 3) * 8), sb = __shfl_sync(0xffffffffu, some[1], (lane & 3) * 8);
        bool fails = false;
        if (lane < 8) {
          const int x = lane & 4 ? xb : xa, any = lane & 4 ? sb : sa, ef = x & 0x7FF00000, row = row0 + lane;
          const bool wild = (x | any) != 0 && (ef < (123 << 20) || ef > (1923 << 20));
          // scale (exponent) and factors of the drains at it, or one below or above
          int4 state = dn ? sR[row] : make_int4(0, -1, -1, 0);
          if (ef != 0 && (state.x == 0 || ef >= state.x - (1 << 20))) {
            const bool fresh = state.x == 0 || ef > state.x + (1 << 20);
            state.y = (int)(lo | (fresh ? 0u : (uint32_t)state.y));
            state.z = (int)(hi | (fresh ? 0u : (uint32_t)state.z));
            state.x = fresh ? ef : state.x;
          }
          if (dn + 1 < ndrains) sR[row] = state;
          constexpr uint64_t all = (1ull << K) - 1;
          const uint64_t good = ((uint64_t)(uint32_t)state.z << 32 | (uint32_t)state.y) & all;
          fails = dn + 1 == ndrains && good != all;
          sX[r * BM + row] = wild || fails ? CELL_PLAIN : ef - (1022 << 20);
          fails = fails && !wild;
        }
        const uint32_t f = __ballot_sync(0xffffffffu, fails);
        if (f != 0u && (f & (f - 1)) == 0u) {  // one of eight rows: here and now; more of them are many, for the epilogue's lanes
          const int row = row0 + __ffs(f) - 1;
          whole_cell<FORM, D>(p, t * BM + row);
          if (lane == 0) sX[r * BM + row] = CELL_DONE;
        }
        __syncwarp();
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(xfull + 8 * r);
    }
  } else if (warp == G_WARPS - 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      const uint32_t a0 = smem_u32(sS), b0 = a0 + G_ASTAGE;
      uint32_t n = 0, dr = 0, tile = 0;  // parts, drains, tiles
      bool ok = true;
      for (int64_t t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++tile) {
        for (int part = 0; part < nparts; ++part, ++n) {
          const uint32_t buf = dr % BUFS;
          const bool first = part % G_DRAIN == 0;
          if (first && !mbar_wait(tempty + 8 * buf, ((dr / BUFS) & 1u) ^ 1u, p.err)) { ok = false; break; }
          const int st = n % AF::STAGES;
          if (!mbar_wait(full + 8 * st, (n / AF::STAGES) & 1u, p.err)) { ok = false; break; }
          tc_fence_after();
          const uint64_t ad = f_desc(a0 + (uint32_t)(st * AF::STAGE), BM * 16);
          const uint64_t bd = f_desc(b0 + (uint32_t)(st * AF::STAGE), G_ND * NC * 16);
          const uint32_t d0 = tmem + buf * (G_ND * NC);
          // Digits p and p + 1 of the cells, interleaved, against T's rows (T_e, T_(e-1)) of e = 0 .. 7 - p at once:
          // their blocks of NC rows follow one another as the columns of the orders p .. 7 do. Wide MMAs because
          // one takes 45 cycles at any N <= 64 (in two above 256 columns).
#pragma unroll
          for (int P = 0; P < G_ND / 2; ++P)
#pragma unroll
            for (int c = 0; c < G_CH; c += 2) {
              constexpr int most = 256 / NC * NC;
              const int cols = (G_ND - 2 * P) * NC, n0 = cols < most ? cols : most;
              const uint32_t acc = first && P == 0 && c == 0 ? 0u : 1u;
              const uint64_t a = ad + (P * G_CH + c) * BM, b = bd + c * (G_ND * NC);
              mma<false>(d0 + 2 * P * NC, a, b, make_idesc(0, BM, n0), acc);
              if (cols > n0) mma<false>(d0 + 2 * P * NC + n0, a, b + n0, make_idesc(0, BM, cols - n0), acc);
            }
          tc_commit(empty + 8 * st);
          if (part == nparts - 1 || part % G_DRAIN == G_DRAIN - 1) {
            tc_commit(tfull + 16 * (tile & 1u) + 8 * buf);
            ++dr;
          }
        }
      }
      tc_commit(smem_u32(&bars->done));
      mbar_wait(smem_u32(&bars->done), 0, p.err);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue: one cell per thread, two sets of warps on alternate tiles ----------------
    const int q = warp & 3, set = warp >> 2;
    const uint32_t lanes = (uint32_t)(q * 32) << 16;
    int64_t i = set;
    uint32_t phases = 0;  // of this set's two barriers: a set waits for each of its drains, in order
    bool ok = true;
    for (int64_t t = blockIdx.x + (int64_t)set * gridDim.x; t < ntiles && ok; t += 2 * (int64_t)gridDim.x, i += 2) {
      const int64_t e = t * BM + q * 32 + lane;
      const bool live = e < p.ncells;
      int vid[NV], cid[NV];
      bool bad = false;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        vid[v] = live ? __ldg(p.c2v + e * NV + v) : 0;
        cid[v] = 0;
        if (live && p.validate && (vid[v] < 0 || vid[v] >= p.nverts)) bad = true;
        if constexpr (FORM == FORM_ADVDIFF) {
          cid[v] = live ? __ldg(p.c2d + e * NV + v) : 0;
          if (live && p.validate && (cid[v] < 0 || cid[v] >= p.ncoefnodes)) bad = true;
        }
      }
      const bool work = live && !bad;
      double X[NV][D];
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int r = 0; r < D; ++r) X[v][r] = work ? __ldg(p.coords + (int64_t)vid[v] * D + r) : 0.0;
      double Gb[K];
      bool wild = false, done = false;
      for (int dn = 0; dn < ndrains; ++dn) {
        const uint32_t dr = (uint32_t)(i * ndrains + dn), buf = dr % BUFS;
        if (!mbar_wait(tfull + 16 * set + 8 * buf, (phases >> buf) & 1u, p.err)) { ok = false; break; }
        phases ^= 1u << buf;
        __syncwarp();
        tc_fence_after();
        const int x20 = sX[(dr % G_XRING) * BM + q * 32 + lane];
        wild = wild || x20 == CELL_PLAIN;
        done = x20 == CELL_DONE;
        __syncwarp();
        if (lane == 0) mbar_arrive(xempty + 8 * (int)(dr % G_XRING));
#pragma unroll
        for (int k0 = 0; k0 < K; k0 += 4) {
          uint32_t v[G_ND][4];
#pragma unroll
          for (int d = 0; d < G_ND; ++d) tmem_ld4(tmem + lanes + buf * (G_ND * NC) + d * NC + k0, v[d]);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (k0 + j < K) {
              int w[G_ND];
#pragma unroll
              for (int d = 0; d < G_ND; ++d) w[d] = __float2int_rn(__uint_as_float(v[d][j]));
              // sum_d w_d 2^(43 - 8 d): the last two orders rounded
              const int64_t x = ((int64_t)w[0] << G_SH) + ((int64_t)w[1] << (G_SH - 8)) + ((int64_t)w[2] << (G_SH - 16)) +
                                ((int64_t)w[3] << (G_SH - 24)) + ((int64_t)w[4] << (G_SH - 32)) +
                                ((w[5] << 3) + ((w[6] + 16) >> 5) + ((w[7] + 4096) >> 13));
              const double a = from_fixed_any((uint32_t)(x >> 32), (uint32_t)x, (uint32_t)(x20 + __ldg(p.kexp20 + k0 + j)));
              Gb[k0 + j] = dn == 0 ? a : Gb[k0 + j] + a;
            }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty + 8 * buf);
      }
      if (!ok) break;
      if (live && bad) {
        atomicOr(p.err, ERR_INDEX);
        if (p.local)
          for (int j = 0; j < NL; ++j) p.local[e * NL + j] = 0.0;
      }
      if (work && !done) {
        if (wild) {
          double tmp[K];
          plain_gbar<FORM, D>(p, e, tmp);
#pragma unroll
          for (int k = 0; k < K; ++k) Gb[k] = tmp[k];
        }
        finish_cell<FORM, D>(p, e, vid, cid, X, Gb);
      }
      __syncwarp();
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == G_WARPS - 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(bars->tmem_base), "r"(TMEM_COLS)
                 : "memory");
  }
}

template <int FORM, int D>
cudaError_t launch_adj(const BwdParams& p, int num_sms, cudaStream_t s) {
  constexpr int fixed = Adj<FORM, D>::STAGES * Adj<FORM, D>::STAGE + G_XRING * BM * 4 + G_SCAN * 8 * 16 + BM * 16 + (int)sizeof(GBars) + 64;
  static_assert(fixed + 11 * Adj<FORM, D>::K * 16 <= 227 * 1024, "P4 tetrahedra have the most drains, 11");
  const int ndrains = ((p.N + G_PE - 1) / G_PE + G_DRAIN - 1) / G_DRAIN, smem = fixed + ndrains * Adj<FORM, D>::K * 16;
  const int grid = (int)std::min<int64_t>((p.ncells + BM - 1) / BM, num_sms);
  auto kern = k_backward_tc<FORM, D>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, G_THREADS, smem, s>>>(p);
  return cudaGetLastError();
}

template <int FORM, int D>
void adj_image(int degree, int cell, std::vector<uint8_t>& img, BwdImage& h) {
  std::vector<int32_t>& kexp20 = h.kexp20;
  using AF = Adj<FORM, D>;
  const int ns = nnodes(cell, degree), N = ns * ns, nparts = (N + G_PE - 1) / G_PE;
  std::vector<double> T;
  reference_tensor(FORM, degree, cell, T);
  img.assign((size_t)nparts * AF::TSTAGE, 0);
  kexp20.assign(AF::K, 0);
  const int len = G_DRAIN * G_PE, ndrains = (N + len - 1) / len;
  h.large.assign((size_t)2 * ndrains * AF::K * 4, 0);
  h.rows.assign((size_t)N * AF::KP, 0.0);
  for (int k = 0; k < AF::K; ++k) {
    double big = 0.0;
    for (int o = 0; o < N; ++o) big = std::max(big, std::fabs(T[(size_t)k * N + o]));
    for (int o = 0; o < N; ++o) {
      h.rows[(size_t)o * AF::KP + k] = T[(size_t)k * N + o];
      if (std::fabs(T[(size_t)k * N + o]) < std::ldexp(big, -G_WEAK_T)) continue;
      for (int v = 0; v < 2; ++v) {
        const int bit = mask_bit(o % len, v == 0);
        h.large[((size_t)(v * ndrains + o / len) * AF::K + k) * 4 + bit / 32] |= 1u << (bit % 32);
      }
    }
    int y = 0;
    if (big > 0) std::frexp(big, &y);
    kexp20[k] = (y - 12 - G_SH + 1054) * (1 << 20);  // order 0: leading digits of 2^-6 each, 2^43 in the sum
    for (int o = 0; o < N; ++o) {
      const uint64_t U = (uint64_t)(int64_t)std::nearbyint(std::ldexp(T[(size_t)k * N + o], G_FB - y)) + G_BIAS;
      uint8_t* part = img.data() + (size_t)(o / G_PE) * AF::TSTAGE;
      for (int e = 0; e < G_ND; ++e)
        for (int w = 0; w < 2; ++w) {  // T_e beside the pair's leading digit, T_(e-1) beside the other
          const int q = e - w;
          const uint16_t h = q < 0 ? 0 : half_of_int((int)((U >> (8 * (G_ND - 1 - q))) & 0xFF) - 128);
          std::memcpy(part + (size_t)((o % G_PE / 4 * G_ND + e) * AF::NC + k) * 16 + (o % 4) * 4 + w * 2, &h, 2);
        }
    }
  }
}

}  // namespace

// Where this kernel runs instead of the plain one: where it is the faster (us for 196,608 cells of random dA, this / plain).
// Advection-diffusion everywhere: triangles P1 84 / 111 to P4 379 / 1230, tetrahedra P1 221 / 362, P2 206 / 1400, P3 670 /
// 5100; Helmholtz on tetrahedra, P1 104 / 114 to P3 408 / 1066, and on triangles P2 76 / 85 and P3 118 / 185,
// but not P1 (54 / 51) and P4 (380 / 371: 225 entries, rows that only 8-byte loads can take). The mass matrix
// has one FMA an entry, which the FP64 pipe does as fast as its 2 x 8 bytes are read (tetrahedra P2 125 / 91).
int backward_tc_use(int form, int degree, int cell) {
  if (form == FORM_HELMHOLTZ) return cell == CELL_TET || degree == 2 || degree == 3;
  return form == FORM_ADVDIFF;
}

void build_backward_image(int form, int degree, int cell, std::vector<uint8_t>& img, BwdImage& h) {
  const bool tri = cell == CELL_TRI;
  if (form == FORM_HELMHOLTZ)
    tri ? adj_image<FORM_HELMHOLTZ, 2>(degree, cell, img, h) : adj_image<FORM_HELMHOLTZ, 3>(degree, cell, img, h);
  else tri ? adj_image<FORM_ADVDIFF, 2>(degree, cell, img, h) : adj_image<FORM_ADVDIFF, 3>(degree, cell, img, h);
}

int launch_backward_tc(int form, int cell, const BwdParams& p, int num_sms, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool tri = cell == CELL_TRI;
  switch (form) {
    case FORM_HELMHOLTZ:
      return (int)(tri ? launch_adj<FORM_HELMHOLTZ, 2>(p, num_sms, s) : launch_adj<FORM_HELMHOLTZ, 3>(p, num_sms, s));
    case FORM_ADVDIFF:
      return (int)(tri ? launch_adj<FORM_ADVDIFF, 2>(p, num_sms, s) : launch_adj<FORM_ADVDIFF, 3>(p, num_sms, s));
  }
  return (int)cudaErrorInvalidValue;
}

}  // namespace coffee
