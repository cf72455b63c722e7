// tcgen05 local assembly of HELMHOLTZ and ADVDIFF on prisms in split tf32 with the quadrature summed in two steps.
//
// Contracted over all points at once (k_prism_tc.cu) an element matrix takes K = 7 (k+2)^3 columns against
// ((k+1)^2 (k+2) / 2)^2 outputs: 8.9 MFLOP of split-tf32 MMAs a P3 cell, whose 13 slices also need the factors
// formed five times over. But points and basis are products of triangle and interval, phi = psi(s,t) zeta(z), so
// the producers first sum the factors over z, per triangle point qt and pair (iz, jz), into eight fields,
//   x0 = m zz + V_zz z'z' (+ beta_z z z')          x4 = V_sz z z'    x5 = V_sz z' z (+ beta_s z z)
//   x1, x2, x3 = V_ss, V_st, V_tt zz               x6 = V_tz z z'    x7 = V_tz z' z (+ beta_t z z)
// (zz = zeta_iz zeta_jz and so on), and the MMA contracts those over qt with the eight products of psi_it, psi_jt
// and their derivatives: K = 8 (k+2)^2 columns, one row per (cell, z pair), nt^2 outputs a row: 1.5 MFLOP a P3
// cell, and each factor is formed once.
// As in k_prism_tc.cu the sums are taken about the cell's factors g_c at the centre of the reference prism:
// fields of w_q (g(x_q) - g_c) first, then one more "point" with the fields of g_c against the products summed
// with the triangle's weights, so that the accumulator stays small while it is added to most often.
//
// Only TF32X3: the other precisions are defined by the parts that each point's factors are held in, and sums over z
// rounded to those parts are other numbers (TF32 here and there: 3e-4 of the entries apart).
// Bound by shared memory (L1 data pipe 72 % busy beside the MMAs' operands, 78 of 7.5 KB a P3 tile) and, with it, the
// latency of the fields' and the epilogue's chains: a seventh fewer wavefronts by padding gained 2 % at P3, lost 3 % at P1.
// Factors and fields are separate warps, two tiles of factors in flight, because in the same warps one after the other
// they took 24,000 cycles a P3 tile (15,400 now); matrix rows put
// together in shared memory because stores of a thread's own runs of nt entries touch 32 sectors each (P4: 48,000
// cycles a tile of stores, 22,000 now).
//
// Rows (M = 128 TMEM lanes): CPW cells times NR z pairs in each lane quadrant, iz <= jz for HELMHOLTZ (symmetric:
// the pair's block is also written transposed), all pairs for ADVDIFF. Columns: nt^2 outputs (9, 36, 100, 225).
//   warps 0-3    epilogue: a thread has one (cell, z pair); matrix rows are put together in shared memory
//   warps 4-11   fields, chunk by chunk into the A operand
//   warp 12      MMA issue
//   warp 13      the table's chunks, one bulk copy each
//   warps 14-15  gather, a tile each in turn (bilinear coefficients, (eps, b), factors at the centre)
//   warps 16-19  factors at the points of the next tile
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cstdint>
#include <cstring>
#include "coffee_internal.h"
#include "tc_common.cuh"
#include "prism_common.cuh"

namespace coffee {
namespace {

using namespace tc;

constexpr int Z_FIELD0 = 4, Z_NFIELD = 256, Z_LOADER = 13, Z_GATHER = 14, Z_FACT0 = 16, Z_NFACT = 128;
constexpr int Z_THREADS = 20 * 32;
constexpr int Z_CB = 64, Z_QC = 2;  // bytes of a row in one K chunk: 8 fields of 2 triangle points
constexpr int Z_TP = 2, Z_GP = 2;   // split-tf32 parts of table and fields
constexpr int Z_MAX_STAGES = 6;
constexpr int Z_NREC = 4;   // tiles of cell records
constexpr int Z_REC = 64;   // floats of a cell's record: A..G [7][3], (eps, b) [6][4], factors at the centre [9], live

template <int FORM, int DEG>
struct Zs {
  static constexpr bool sym = FORM == FORM_HELMHOLTZ;
  static constexpr int KQ = sym ? 7 : 9, P = DEG + 2, QT = P * P, QZ = P, Q = QT * QZ;
  static constexpr int NT = (DEG + 1) * (DEG + 2) / 2, NZ = DEG + 1, n = NT * NZ;
  static constexpr int NR = sym ? NZ * (NZ + 1) / 2 : NZ * NZ;    // rows of a cell
  static constexpr int CPW = 32 / NR, CT = 4 * CPW;               // cells of a lane quadrant, of a tile
  // Rows of one cell a field thread forms (z pairs j and j + HR): its factors are read once for both, 4,200 -> 2,100
  // cycles of shared-memory reads a P3 tile (Helmholtz P3 262 -> 237 us, advection-diffusion P2 354 -> 316). Not P1,
  // whose ten cells a quadrant would not fit sixteen threads, nor P4, which has two stages only (see ZLayout).
  static constexpr int RPT = DEG == 2 || DEG == 3 ? 2 : 1, HR = (NR + RPT - 1) / RPT;
  static_assert(RPT == 1 || CPW * HR <= 16, "sixteen threads a lane quadrant");
  static constexpr int NO = NT * NT, NP = (NO + 15) / 16 * 16;
  static constexpr int FS = sym ? 8 : 12;                         // floats of a point's factors in shared memory
  static constexpr int CS = Q * FS + (36 - Q * FS % 32) % 32;     // of a cell's: cells start 4 banks apart
  static constexpr int NKC = (QT + 1 + Z_QC - 1) / Z_QC;          // K chunks
  static constexpr int A = Z_GP * BM * Z_CB, B = Z_TP * NP * Z_CB, STAGE = A + B;
};

struct alignas(8) ZBars {
  uint64_t full[Z_MAX_STAGES], empty[Z_MAX_STAGES], tfull[2], tempty[2], cfull[Z_NREC], cempty[Z_NREC], ffull[2], fempty[2];
  uint64_t done;
  uint32_t tmem_base;
};

template <int FORM, int DEG>
struct ZLayout : Zs<FORM, DEG> {
  using S = Zs<FORM, DEG>;
  static constexpr int OUTS = S::CPW * S::NZ * S::n;  // floats of a quadrant's matrix rows of one it
  static constexpr int FIXED = (2 * S::CT * S::CS + Z_NREC * S::CT * Z_REC + (4 * OUTS + 3) / 4 * 4) * 4 + (int)sizeof(ZBars);
  static constexpr int fit = (227 * 1024 - FIXED) / S::STAGE;
  static constexpr int NST = fit < Z_MAX_STAGES ? fit : Z_MAX_STAGES;
  static constexpr int SMEM = NST * S::STAGE + FIXED;
  // RPT = 2: a thread waits for the slots of every other chunk, k' = k - 2 or, from one tile to the next, k - 3 before
  // k. That chunk k' - NST was consumed tells it that chunk k - 2 NST was, and with it which of the slot's two phases the
  // parity means, only if k - k' <= NST.
  static_assert(NST >= (S::RPT == 2 ? 3 : 2), "stages");
};

__device__ __forceinline__ void tmem_ld1(uint32_t taddr, uint32_t* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(v[0]) : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, uint32_t* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
}
template <int N>
__device__ __forceinline__ void tmem_row(uint32_t taddr, uint32_t (&v)[N]) {  // N consecutive columns
  static_assert(N < 16, "up to 15 columns");
  if constexpr (N & 8) tmem_ld8(taddr, v);
  if constexpr (N & 4) tmem_ld4(taddr + (N & 8), v + (N & 8));
  if constexpr (N & 2) tmem_ld2(taddr + (N & 12), v + (N & 12));
  if constexpr (N & 1) tmem_ld1(taddr + (N & 14), v + (N & 14));
}

// A cell's bilinear coefficients and (eps, b), of its record
template <int KQ>
struct Cell {
  float JA[3], JB[3], JC[3], JD[3], JE[3], JF[3], JG[3], CF[6][4];
  __device__ __forceinline__ void load(const float* rec) {
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      JA[r] = rec[r]; JB[r] = rec[3 + r]; JC[r] = rec[6 + r]; JD[r] = rec[9 + r];
      JE[r] = rec[12 + r]; JF[r] = rec[15 + r]; JG[r] = rec[18 + r];
    }
#pragma unroll
    for (int v = 0; v < 6; ++v)
#pragma unroll
      for (int c = 0; c < 4; ++c) CF[v][c] = KQ == 9 ? rec[21 + v * 4 + c] : 0.f;
  }
  __device__ __forceinline__ void factors(const float4 pq, float (&g)[9]) const {
    prism_point_factors<KQ>(pq, JA, JB, JC, JD, JE, JF, JG, CF, g);
  }
};

// x += the fields of one z point with products w = (zz, zz', z'z, z'z') from factors g (m, V.. or V.., beta)
template <bool SYM>
__device__ __forceinline__ void add_fields(const float* g, const float4 w, float (&x)[8]) {
  const float* V = SYM ? g + 1 : g;  // ss, st, sz, tt, tz, zz
  x[0] = SYM ? fmaf(g[0], w.x, fmaf(V[5], w.w, x[0])) : fmaf(g[8], w.y, fmaf(V[5], w.w, x[0]));
  x[1] = fmaf(V[0], w.x, x[1]);
  x[2] = fmaf(V[1], w.x, x[2]);
  x[3] = fmaf(V[3], w.x, x[3]);
  x[4] = fmaf(V[2], w.y, x[4]);
  x[5] = fmaf(V[2], w.z, SYM ? x[5] : fmaf(g[6], w.x, x[5]));
  x[6] = fmaf(V[4], w.y, x[6]);
  x[7] = fmaf(V[4], w.z, SYM ? x[7] : fmaf(g[7], w.x, x[7]));
}

template <int FORM, int DEG>
__global__ void __launch_bounds__(Z_THREADS, 1) k_prism_sum_tc(const TcParams p) {
  using S = Zs<FORM, DEG>;
  using L = ZLayout<FORM, DEG>;
  constexpr int NKC = S::NKC, NST = L::NST, QT = S::QT, QZ = S::QZ, Q = S::Q, NT = S::NT, NZ = S::NZ, n = S::n, NR = S::NR,
                CPW = S::CPW, CT = S::CT, NP = S::NP, FS = S::FS, CS = S::CS, KQ = S::KQ;
  extern __shared__ __align__(1024) uint8_t smem[];
  float* sF = reinterpret_cast<float*>(smem + NST * L::STAGE);  // [2][CT][CS]
  float* sC = sF + 2 * CT * CS;                                 // [Z_NREC][CT][Z_REC]
  float* sO = sC + Z_NREC * CT * Z_REC;                         // [4][OUTS]
  ZBars* bars = reinterpret_cast<ZBars*>(sO + (4 * L::OUTS + 3) / 4 * 4);
  const float4* ztab = reinterpret_cast<const float4*>(p.image + (size_t)NKC * L::B);  // [QZ + 1][NR]
  const float4* points = ztab + (QZ + 1) * NR;                                          // [Q] (s, t, z, weight)

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int64_t ntiles = (p.ncells + CT - 1) / CT;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(smem_u32(&bars->full[s]), Z_NFIELD / S::RPT + 1);
      mbar_init(smem_u32(&bars->empty[s]), 1);
    }
    for (int r = 0; r < 2; ++r) {
      mbar_init(smem_u32(&bars->tfull[r]), 1);
      mbar_init(smem_u32(&bars->tempty[r]), EPI_WARPS);
      mbar_init(smem_u32(&bars->ffull[r]), Z_NFACT);
      mbar_init(smem_u32(&bars->fempty[r]), Z_NFIELD);
    }
    for (int r = 0; r < Z_NREC; ++r) {
      mbar_init(smem_u32(&bars->cfull[r]), 32);
      mbar_init(smem_u32(&bars->cempty[r]), Z_NFIELD);  // fields are the last to read a record
    }
    mbar_init(smem_u32(&bars->done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == MMA_WARP) {
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

  if (warp >= Z_FACT0) {
    // ---------------- factors: TPC threads share a cell's points ----------------
    constexpr int TPC = Z_NFACT / CT;
    const int id = threadIdx.x - Z_FACT0 * 32, cell = id / TPC, q0 = id % TPC;
    uint32_t i = 0;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x, ++i) {
      const uint32_t f = i & 1u, r = i % Z_NREC;
      if (!mbar_wait(smem_u32(&bars->cfull[r]), (i / Z_NREC) & 1u, p.err)) break;
      if (!mbar_wait(smem_u32(&bars->fempty[f]), ((i >> 1) & 1u) ^ 1u, p.err)) break;
      if (cell < CT) {
        const float* rec = sC + (r * CT + cell) * Z_REC;
        float* o = sF + (f * CT + cell) * CS;
        float c[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) c[k] = rec[45 + k];
        if (rec[54] != 0.f) {
          Cell<KQ> J;
          J.load(rec);
          for (int q = q0; q < Q; q += TPC) {
            const float4 pq = __ldg(points + q);
            float g[12] = {}, h[9];
            J.factors(pq, h);
#pragma unroll
            for (int k = 0; k < KQ; ++k) g[k] = fmaf(-pq.w, c[k], h[k]);
#pragma unroll
            for (int v = 0; v < FS / 4; ++v)
              *reinterpret_cast<float4*>(o + q * FS + 4 * v) = make_float4(g[4 * v], g[4 * v + 1], g[4 * v + 2], g[4 * v + 3]);
          }
        } else {
          for (int q = q0; q < Q; q += TPC)
#pragma unroll
            for (int v = 0; v < FS / 4; ++v) *reinterpret_cast<float4*>(o + q * FS + 4 * v) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
      mbar_arrive(smem_u32(&bars->ffull[f]));
    }
  } else if (warp >= Z_FIELD0 && warp < MMA_WARP) {
    // ---------------- fields: RPT (cell, z pair) rows per thread, one of a chunk's two triangle points ----------------
    // RPT = 1: two chunks at once, 128 rows x 2 points; RPT = 2: each half of the warps every other chunk
    constexpr int RPT = S::RPT, HR = S::HR, LANES = BM / RPT, UC = 3 - RPT;
    const int id = threadIdx.x - Z_FIELD0 * 32, at = id % LANES, sub = id / LANES & 1, half = RPT == 2 ? id >> 7 : 0;
    const int q = at / (32 / RPT), l = at % (32 / RPT), cw = l % CPW, j = l / CPW;
    const bool used = j < HR;
    const int cl = q * CPW + cw;
    float4 w[RPT][QZ];
#pragma unroll
    for (int y = 0; y < RPT; ++y)
#pragma unroll
      for (int z = 0; z < QZ; ++z) w[y][z] = __ldg(ztab + z * NR + (j + y * HR < NR ? j + y * HR : 0));
    uint32_t c = 0, i = 0;
    bool ok = true;
    for (int64_t t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++i, c += NKC) {
      const uint32_t f = i & 1u, r = i % Z_NREC;
      // the record: its words are written before the factors that ffull stands for
      if (!mbar_wait(smem_u32(&bars->cfull[r]), (i / Z_NREC) & 1u, p.err)) break;
      if (!mbar_wait(smem_u32(&bars->ffull[f]), (i >> 1) & 1u, p.err)) break;
      const float* F = sF + (f * CT + cl) * CS;
      for (int kc = half; kc < NKC && ok; kc += 2) {
        float x[UC][RPT][8] = {};
#pragma unroll
        for (int u = 0; u < UC; ++u) {
          const int qt = (kc + u) * Z_QC + sub;
          if (used && qt < QT) {
            const float4* f4 = reinterpret_cast<const float4*>(F + qt * QZ * FS);
#pragma unroll
            for (int z = 0; z < QZ; ++z) {
              float g[FS];
#pragma unroll
              for (int v = 0; v < FS / 4; ++v) *reinterpret_cast<float4*>(g + 4 * v) = f4[z * (FS / 4) + v];
#pragma unroll
              for (int y = 0; y < RPT; ++y) add_fields<S::sym>(g, w[y][z], x[u][y]);
            }
          } else if (used && qt == QT) {
#pragma unroll
            for (int y = 0; y < RPT; ++y)
              add_fields<S::sym>(sC + (r * CT + cl) * Z_REC + 45, __ldg(ztab + QZ * NR + (j + y * HR < NR ? j + y * HR : 0)), x[u][y]);
          }
        }
#pragma unroll
        for (int u = 0; u < UC; ++u) {
          if (kc + u >= NKC) break;
          const uint32_t k = c + kc + u;
          const int s = (int)(k % NST);
          if (!mbar_wait(empty + 8 * s, ((k / NST) & 1u) ^ 1u, p.err)) { ok = false; break; }
          uint8_t* a = smem + (size_t)s * L::STAGE;
#pragma unroll
          for (int y = 0; y < RPT; ++y) {
            // (the rows past the cells', which RPT = 2 leaves as they are, feed accumulator rows that nothing reads)
            const int zi = j + y * HR, row = q * 32 + zi * CPW + cw;
            if (RPT == 1 || (used && zi < NR)) {
              store_unit<true, Z_GP>(a + canon_off(row, sub * 32, Z_CB), BM * Z_CB, &x[u][y][0]);
              store_unit<true, Z_GP>(a + canon_off(row, sub * 32 + 16, Z_CB), BM * Z_CB, &x[u][y][4]);
            }
          }
          fence_proxy_async();
          mbar_arrive(full + 8 * s);
        }
      }
      if (!ok) break;
      mbar_arrive(smem_u32(&bars->fempty[f]));
      mbar_arrive(smem_u32(&bars->cempty[r]));
    }
  } else if (warp >= Z_GATHER) {
    // ---------------- cells, two tiles in flight ----------------
    uint32_t i = warp - Z_GATHER;
    int nv[6], nc[6];  // the indices of the cell after this one, requested a cell ahead
    auto request = [&](int64_t e) {
#pragma unroll
      for (int v = 0; v < 6; ++v) {
        nv[v] = e < p.ncells ? __ldg(p.c2v + e * 6 + v) : 0;
        nc[v] = KQ == 9 && e < p.ncells ? __ldg(p.c2d + e * 6 + v) : 0;
      }
    };
    request((blockIdx.x + (int64_t)i * gridDim.x) * CT + lane);
    for (int64_t t = blockIdx.x + (int64_t)i * gridDim.x; t < ntiles; t += 2 * (int64_t)gridDim.x, i += 2) {
      const uint32_t r = i % Z_NREC;
      if (!mbar_wait(smem_u32(&bars->cempty[r]), ((i / Z_NREC) & 1u) ^ 1u, p.err)) break;
      for (int l = lane; l < CT; l += 32) {
        const int64_t e = t * CT + l;
        float* rec = sC + (r * CT + l) * Z_REC;
        bool live = e < p.ncells, bad = false;
        int vid[6], cid[6];
#pragma unroll
        for (int v = 0; v < 6; ++v) {
          vid[v] = nv[v];
          cid[v] = nc[v];
          if (p.validate && live && (vid[v] < 0 || vid[v] >= p.nverts)) bad = true;
          if (KQ == 9 && p.validate && live && (cid[v] < 0 || cid[v] >= p.ncoefnodes)) bad = true;
        }
        request(l + 32 < CT ? e + 32 : (t + 2 * (int64_t)gridDim.x) * CT + lane);
        if (bad) {
          atomicOr(p.err, ERR_INDEX);
          live = false;
        }
        float g[9] = {};
        if (live) {
          Cell<KQ> J;
          if constexpr (KQ == 9) coef_rows<6, 4>(p, cid, J.CF);
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            double X[6];
#pragma unroll
            for (int v = 0; v < 6; ++v) X[v] = __ldg(p.coords + (int64_t)vid[v] * 3 + k);
            // J is bilinear: d/ds = A + z B, d/dt = C + z D, d/dz = E + s F + t G, differences taken in FP64
            const double b1 = X[1] - X[0], b2 = X[2] - X[0], t1 = X[4] - X[3], t2 = X[5] - X[3];
            const double h0 = X[3] - X[0], h1 = X[4] - X[1], h2 = X[5] - X[2];
            J.JA[k] = (float)b1;
            J.JB[k] = (float)(t1 - b1);
            J.JC[k] = (float)b2;
            J.JD[k] = (float)(t2 - b2);
            J.JE[k] = (float)h0;
            J.JF[k] = (float)(h1 - h0);
            J.JG[k] = (float)(h2 - h0);
          }
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            rec[k] = J.JA[k]; rec[3 + k] = J.JB[k]; rec[6 + k] = J.JC[k]; rec[9 + k] = J.JD[k];
            rec[12 + k] = J.JE[k]; rec[15 + k] = J.JF[k]; rec[18 + k] = J.JG[k];
          }
          if constexpr (KQ == 9) {
#pragma unroll
            for (int v = 0; v < 6; ++v)
#pragma unroll
              for (int k = 0; k < 4; ++k) rec[21 + v * 4 + k] = J.CF[v][k];
          }
          J.factors(make_float4(1.f / 3.f, 1.f / 3.f, 0.5f, 1.f), g);
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) rec[45 + k] = g[k];
        rec[54] = live ? 1.f : 0.f;
      }
      mbar_arrive(smem_u32(&bars->cfull[r]));
    }
  } else if (warp == Z_LOADER) {
    // ---------------- the table, chunk by chunk ----------------
    if (lane == 0) {
      uint32_t c = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < ntiles && ok; t += gridDim.x)
        for (int kc = 0; kc < NKC; ++kc, ++c) {
          const int s = (int)(c % NST);
          if (!mbar_wait(empty + 8 * s, ((c / NST) & 1u) ^ 1u, p.err)) { ok = false; break; }
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full + 8 * s), "r"((uint32_t)L::B)
                       : "memory");
          asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                           smem_u32(smem + (size_t)s * L::STAGE + L::A)),
                       "l"(p.image + (size_t)kc * L::B), "r"((uint32_t)L::B), "r"(full + 8 * s)
                       : "memory");
        }
      // no copy may land after this block has left: wait for the last chunk of each stage
      for (uint32_t k = c > (uint32_t)NST ? c - NST : 0; k < c; ++k) mbar_wait(full + 8 * (k % NST), (k / NST) & 1u, p.err);
    }
    __syncwarp();
  } else if (warp == MMA_WARP) {
    // ---------------- MMA issuer: D[row][output] += fields . table ----------------
    if (lane == 0) {
      using PS = Passes<PREC_TF32X3>;
      const uint32_t s0 = smem_u32(smem), idesc = make_idesc(2, BM, NP);
      uint32_t c = 0, i = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++i) {
        const uint32_t buf = i & 1u;
        if (!mbar_wait(smem_u32(&bars->tempty[buf]), ((i >> 1) & 1u) ^ 1u, p.err)) break;
        tc_fence_after();
        for (int kc = 0; kc < NKC; ++kc, ++c) {
          const int s = (int)(c % NST);
          if (!mbar_wait(full + 8 * s, (c / NST) & 1u, p.err)) { ok = false; break; }
          tc_fence_after();
          const uint64_t a = make_desc(s0 + s * L::STAGE, 8 * Z_CB), b = make_desc(s0 + s * L::STAGE + L::A, 8 * Z_CB);
#pragma unroll
          for (int ks = 0; ks < Z_CB / 32; ++ks)
#pragma unroll
            for (int x = 0; x < PS::N; ++x)  // descriptor addresses count 16 bytes
              mma<true>(tmem + buf * 256, a + PS::g(x) * (BM * Z_CB / 16) + ks * 16,
                        b + PS::t(x) * (NP * Z_CB / 16) + ks * 16, idesc, (kc | ks | x) ? 1u : 0u);
          tc_commit(empty + 8 * s);
        }
        tc_commit(smem_u32(&bars->tfull[buf]));
      }
      tc_commit(smem_u32(&bars->done));
      mbar_wait(smem_u32(&bars->done), 0, p.err);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue ----------------
    constexpr int VEC = n % 4 == 0 ? 4 : n % 2 == 0 ? 2 : 1;
    const int zi = lane / CPW < NR ? lane / CPW : 0, cw = lane / CPW < NR ? lane % CPW : CPW;
    int iz = zi / NZ, jz = zi % NZ;
    if (S::sym) {
      for (jz = 0; (jz + 1) * (jz + 2) / 2 <= zi;) ++jz;
      iz = zi - jz * (jz + 1) / 2;
    }
    float* st = sO + warp * L::OUTS;
    float* d0 = st + (cw * NZ + iz) * n + jz * NT;  // block (iz, jz) of row it: the columns it NT .. it NT + NT - 1,
    float* d1 = st + (cw * NZ + jz) * n + iz * NT;  // its transpose in (jz, iz): the columns jt, NT + jt, ..
    const bool used = cw < CPW, both = S::sym && used && iz != jz;
    const bool vec = (reinterpret_cast<uintptr_t>(p.out) & (4 * VEC - 1)) == 0;
    constexpr int ITER = VEC > 1 ? (L::OUTS + 32 * VEC - 1) / (32 * VEC) : 1;
    int at[ITER];  // where this lane's vectors of matrix row it = 0 go
#pragma unroll
    for (int x = 0; x < ITER; ++x) {
      const int k = (x * 32 + lane) * VEC, r = k / n;
      at[x] = r / NZ * (n * n) + r % NZ * NT * n + k % n;
    }
    uint32_t i = 0;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x, ++i) {
      const uint32_t buf = i & 1u;
      if (!mbar_wait(smem_u32(&bars->tfull[buf]), (i >> 1) & 1u, p.err)) break;
      __syncwarp();
      tc_fence_after();
      const int64_t e0 = t * CT + warp * CPW, left = p.ncells - e0;
      const int cells = (int)(left < 0 ? 0 : left < CPW ? left : CPW), floats = cells * NZ * n;
      float* A = p.out + e0 * (int64_t)(n * n);
      const uint32_t ta = tmem + ((uint32_t)(warp * 32) << 16) + buf * 256;
#pragma unroll 1
      for (int it = 0; it < NT; ++it) {
        uint32_t v[NT], u[NT];
        tmem_row<NT>(ta + it * NT, v);
        if constexpr (S::sym) {
#pragma unroll
          for (int k = 0; k < NT; ++k) tmem_ld1(ta + k * NT + it, u + k);
        }
        tmem_wait_ld();
        if (used) {
#pragma unroll
          for (int k = 0; k < NT; ++k) d0[k] = __uint_as_float(v[k]);
        }
        if constexpr (S::sym) {
          if (both) {
#pragma unroll
            for (int k = 0; k < NT; ++k) d1[k] = __uint_as_float(u[k]);
          }
        }
        __syncwarp();
        // the quadrant's matrix rows iz NT + it, n contiguous entries each
        if (VEC > 1 && vec) {
#pragma unroll
          for (int x = 0; x < ITER; ++x) {
            const int k = (x * 32 + lane) * VEC;
            if (k < floats) {
              float* dst = A + at[x] + it * n;
              if constexpr (VEC == 4) __stcs(reinterpret_cast<float4*>(dst), *reinterpret_cast<const float4*>(st + k));
              else if constexpr (VEC == 2) __stcs(reinterpret_cast<float2*>(dst), *reinterpret_cast<const float2*>(st + k));
            }
          }
        } else {
#pragma unroll
          for (int cell = 0; cell < CPW; ++cell) {
            if (cell >= cells) break;
#pragma unroll
            for (int z = 0; z < NZ; ++z)
#pragma unroll
              for (int k = 0; k < n; k += 32)
                if (k + lane < n)
                  __stcs(A + (cell * (n * n) + z * NT * n + k) + it * n + lane, st[(cell * NZ + z) * n + k + lane]);
          }
        }
        __syncwarp();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars->tempty[buf]));
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == MMA_WARP) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

template <int FORM, int DEG>
cudaError_t launch_z(const TcParams& p, int num_sms, cudaStream_t s) {
  using L = ZLayout<FORM, DEG>;
  const int64_t ntiles = (p.ncells + L::CT - 1) / L::CT;
  const int grid = (int)(ntiles < num_sms ? ntiles : num_sms);
  const int smem = L::SMEM < 120 * 1024 ? 120 * 1024 : L::SMEM;  // one CTA (one TMEM owner) per SM
  auto kern = k_prism_sum_tc<FORM, DEG>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, Z_THREADS, smem, s>>>(p);
  return cudaGetLastError();
}

template <int FORM>
cudaError_t launch_zd(int degree, const TcParams& p, int num_sms, cudaStream_t s) {
  switch (degree) {
    case 1: return launch_z<FORM, 1>(p, num_sms, s);
    case 2: return launch_z<FORM, 2>(p, num_sms, s);
    case 3: return launch_z<FORM, 3>(p, num_sms, s);
    case 4: return launch_z<FORM, 4>(p, num_sms, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

// TF32X3, both forms at any count. Graph-replayed times, us, one contraction over all points | here:
//   cells                 7           3000          P1 250,000, P2 110,592, P3 55,296, P4 16,000
//   HELMHOLTZ   P1    25 | 10       27 | 13       280 | 148
//               P2    53 | 13       56 | 14       297 | 188
//               P3   441 | 17      436 | 25      1301 | 237
//               P4  2269 | 26     2226 | 55      2231 | 207
//   ADVDIFF     P1    36 | 12       37 | 12       412 | 237
//               P2    75 | 14       77 | 20       417 | 316
//               P3   643 | 17      626 | 32      1871 | 336
//               P4  3306 | 25     3202 | 81      3210 | 381
// The error of one contraction against 64 bits is 1.7-4.8 times this one's.
// MASS (K = (k+2)^3), the CSR forms and the other precisions stay with the other kernel.
bool prism_sum_tc_use(int form, int precision) {
  return (form == FORM_HELMHOLTZ || form == FORM_ADVDIFF) && precision == PREC_TF32X3;
}

// Chunks [chunk][part][NP rows x 64 B canonical] of the table T[o = it nt + jt][qt 8 + f] (after the last point the
// products summed with the triangle's weights), then as floats the z products [QZ + 1][NR][4] (the last row summed
// with z's weights) and the points [QT][QZ][4] (s, t, z, weight).
void build_prism_sum_image(int form, int degree, std::vector<uint8_t>& img) {
  const bool sym = form == FORM_HELMHOLTZ;
  const int p = degree + 2, QT = p * p, nt = (degree + 1) * (degree + 2) / 2, nz = degree + 1;
  const int NO = nt * nt, NP = (NO + 15) / 16 * 16, nkc = (QT + 1 + Z_QC - 1) / Z_QC;
  const int NR = sym ? nz * (nz + 1) / 2 : nz * nz;
  std::vector<double> pts, wts, zp, zw, psi, dpsi, zeta;
  prism_factor_tables(form, degree, pts, wts, psi, dpsi, zp, zw, zeta);
  const size_t part = (size_t)NP * Z_CB, chunk = Z_TP * part;
  img.assign(nkc * chunk, 0);
  for (int it = 0; it < nt; ++it)
    for (int jt = 0; jt < nt; ++jt) {
      double sum[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      for (int qt = 0; qt <= QT; ++qt) {
        double v[8];
        if (qt < QT) {
          const double a = psi[(size_t)qt * nt + it], b = psi[(size_t)qt * nt + jt];
          const double *da = &dpsi[((size_t)qt * nt + it) * 2], *db = &dpsi[((size_t)qt * nt + jt) * 2];
          const double x[8] = {a * b,     da[0] * db[0], da[0] * db[1] + da[1] * db[0], da[1] * db[1],
                               da[0] * b, a * db[0],     da[1] * b,                     a * db[1]};
          for (int f = 0; f < 8; ++f) {
            v[f] = x[f];
            sum[f] += wts[qt] * x[f];
          }
        } else {
          std::memcpy(v, sum, sizeof v);
        }
        for (int f = 0; f < 8; ++f)
          host_store_parts(img.data() + (size_t)(qt / Z_QC) * chunk, part,
                           canon_off(it * nt + jt, (qt % Z_QC * 8 + f) * 4, Z_CB), v[f], true, Z_TP);
      }
    }
  std::vector<float> tail;
  for (int q = 0; q <= p; ++q)
    for (int r = 0; r < NR; ++r) {
      int iz, jz = 0;
      if (sym) {
        while ((jz + 1) * (jz + 2) / 2 <= r) ++jz;
        iz = r - jz * (jz + 1) / 2;
      } else {
        iz = r / nz;
        jz = r % nz;
      }
      double v[4] = {0, 0, 0, 0};
      for (int z = q < p ? q : 0; z < (q < p ? q + 1 : p); ++z) {
        const double *a = &zeta[((size_t)z * nz + iz) * 2], *b = &zeta[((size_t)z * nz + jz) * 2];
        const double w = q < p ? 1.0 : zw[z];
        v[0] += w * a[0] * b[0];
        v[1] += w * a[0] * b[1];
        v[2] += w * a[1] * b[0];
        v[3] += w * a[1] * b[1];
      }
      for (double x : v) tail.push_back((float)x);
    }
  for (int qt = 0; qt < QT; ++qt)
    for (int z = 0; z < p; ++z)
      for (double x : {pts[(size_t)qt * 2], pts[(size_t)qt * 2 + 1], zp[z], wts[qt] * zw[z]}) tail.push_back((float)x);
  const size_t at = img.size();
  img.resize(at + tail.size() * sizeof(float));
  std::memcpy(img.data() + at, tail.data(), tail.size() * sizeof(float));
}

int launch_prism_sum_tc(int form, int degree, const TcParams& p, int num_sms, void* stream) {
  if (p.ncells == 0) return (int)cudaSuccess;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return (int)(form == FORM_HELMHOLTZ ? launch_zd<FORM_HELMHOLTZ>(degree, p, num_sms, s)
                                      : launch_zd<FORM_ADVDIFF>(degree, p, num_sms, s));
}

}  // namespace coffee
