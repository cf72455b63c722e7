// FP64 local and global assembly on the tensor cores: A_e[o] = sum_k G_e[k] T[k][o] with the
// contraction done exactly, in integers, by tcgen05 f16 MMAs.
//
// What bounds the plain FP64 kernel is the FP64 pipe, 2 FMAs per cycle and SM on this GPU: Helmholtz
// P3 on tetrahedra (K = 7 FMAs for each of 400 entries) takes 1400 cycles a cell, ten times the 150
// cycles in which its 3200 bytes reach memory. The f16 MMA does 2000 times the FP64 pipe's products.
// Here every operand is a fixed-point number of FB = 61 or 62 fraction bits, cut into balanced digits
// that an f16 holds exactly:
//
//   G_e[k] 2^tk  = 2^x sum_p g_p 2^(b (ND-1-p) - FB)   per cell one exponent x, |g_p| <= 2^(b-1)
//   T[k][o] 2^-tk = 2^y sum_q t_q 2^(b (ND-1-q) - FB)  per entry one exponent y
//
// (b = 9 with ND = 7 digits for K <= 7 factors, b = 8 with ND = 8 for K <= 36). The products of
// digits with p + q = d have one weight, 2^-bd, so they are contracted together into one accumulator
// per order d < ND: an integer of at most K (d+1) 2^(2b-2) <= 2^22, which FP32 accumulation holds
// exactly. A constant product 4096 x 3072 = 1.5 * 2^23 is contracted along with the digits: with it the
// accumulator lies in [2^23, 2^24), where the float's bit pattern is 0x4B400000 plus the integer, so
// no conversion is needed. (For b = 8 the bound fails for the last order, d = 7, alone: it takes no
// constant and is converted by one FP32 addition.) The epilogue adds the orders in 64-bit integers and
// rounds once to double, again with integer instructions: an entry's error is that rounding plus about
// 2^-56 of max_k |G_k| max_k |T_k|, where K rounded FMAs stood before. Against quadruple precision, rms
// over cells relative to max|A_e|: Helmholtz P3 tetrahedra 2.2e-17 (plain kernel 2.5e-17), advection-
// diffusion P2 4.4e-17 (6.3e-17), and no larger than the plain kernel's for any form, degree and cell.
//
// Operands are K-major without swizzle: 16-byte rows (8 factors of one digit) contiguous in chunks; T by
// 128-entry slice, digit and chunk, the cells by chunk, digit and cell (see the MMA warp for why).
//
// One persistent CTA per SM holds two independent pipelines (halves), which keeps one busy while the
// other waits: in each, three producer warps gather, form the factors in FP64 and store digits, a tile of
// 32 cells each; one warp issues the MMAs (M = 128 entries, N = 32 cells times digits); eight epilogue warps
// (32 entries x 16 cells each) combine the orders in registers and write rows of 32 doubles, 256 bytes. T's digits stay in shared memory where they fit; otherwise the CTAs split
// into groups by 128-entry slices, each with its slices resident, and form the factors once per group.
// What bounds it now is the integer work of the epilogue, about 26 instructions an entry (half of them
// moved to the multiplier pipe, see mad_lo), and the latencies between its phases. 196,608 tetrahedra,
// this kernel / plain: Helmholtz P2 57 / 300 us, P3 158 / 1131 us (0.6 of the copy bandwidth), P4 417 /
// 3310 us; advection-diffusion P2 123 / 1450 us, P4 1.10 / 16.9 ms. Steps on the way (Helmholtz P3): one
// pipeline with 21 warps 479 us; 16 warps of 128 registers 324; multiplications for shifts 311; two
// pipelines 242; 16 cells per epilogue warp, four epilogue warps a scheduler, 169; one wide MMA per digit of T
// instead of one per order and K step 158 (advection-diffusion P2 168 -> 123).
// Cells whose factors are not finite or outside 2^+-900 are evaluated entry by entry in FP64.
#include <cuda_runtime.h>
#include <cuda_fp16.h>
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

constexpr int FN = 32;                 // cells per tile (MMA N)
constexpr int F_HALVES = 2;            // independent pipelines per CTA
constexpr int F_EPI = 8;               // epilogue warps of a half, two per TMEM lane quadrant
constexpr int FC = FN / 2;             // cells per epilogue warp
constexpr int F_PROD = 3;              // producer warps of a half, a tile each in turn
constexpr int F_PWARP0 = F_HALVES * F_EPI, F_MWARP0 = F_PWARP0 + F_HALVES * F_PROD;
constexpr int F_WARPS = F_MWARP0 + F_HALVES;  // 24: six per scheduler, 80 registers a thread
constexpr int F_THREADS = F_WARPS * 32;
constexpr int F_COLS = 256;            // accumulator columns of a half: order d at columns 32 d
constexpr int F_XRING = 8;             // tiles whose cell exponents are kept (operand stages + 2 at least)
constexpr int F_STAGES = 4;            // operand stages of a half at most
constexpr int CELL_SKIP = INT32_MIN, CELL_PLAIN = INT32_MIN + 1;
constexpr uint32_t MAGIC = 0x4B400000u;  // 1.5 * 2^23 as a float

struct alignas(8) FBars {
  uint64_t full[F_HALVES][F_STAGES], empty[F_HALVES][F_STAGES], tfull[F_HALVES], tempty[F_HALVES], done[F_HALVES];
  uint32_t tmem_base;
};

template <int FORM, int D>
struct Digits {
  static constexpr int K = FormK<FORM, D>::value;
  static constexpr int B = FORM == FORM_ADVDIFF ? 8 : 9;   // bits per digit
  static constexpr int ND = FORM == FORM_ADVDIFF ? 8 : 7;  // digits
  static constexpr int FB = FORM == FORM_ADVDIFF ? 62 : 61;  // fraction bits of the fixed-point operands
  static constexpr int KC = (K + 1 + 7) / 8;               // 8-factor chunks per digit, one slot for the constant
  static constexpr int ACH = ND * KC + 1;                  // chunks of a table row, the last one zero
  static constexpr int SLICE = ACH * BM * 16;              // bytes of one 128-entry slice of the table
  static constexpr int STAGE = ND * KC * FN * 16;
  COFFEE_HD static constexpr uint64_t bias() {
    uint64_t s = 0;
    for (int p = 0; p < ND; ++p) s += 1ull << (B - 1 + B * p);
    return s;
  }
};

template <int FORM, int D>
__device__ __noinline__ double plain_entry(const Fp64Params& p, int64_t e, int o) {
  double G[FormK<FORM, D>::value];
  if (!factors64<FORM, D, false>(p, e, G)) return 0.0;
  double acc = 0.0;
#pragma unroll
  for (int k = 0; k < FormK<FORM, D>::value; ++k) acc = fma(G[k], __ldg(p.T + (int64_t)k * p.N + o), acc);
  return acc;
}

// slices: 128-entry slices resident per CTA; groups: CTA groups the slices are split over; nst: operand
// stages of a half
template <int FORM, int D, bool CSR>
__global__ void __launch_bounds__(F_THREADS, 1) k_assemble_fp64_tc(const Fp64Params p, int slices, int groups,
                                                                   int nst) {
  using DG = Digits<FORM, D>;
  constexpr int K = DG::K, KC = DG::KC, ND = DG::ND, B = DG::B;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* sB = smem_raw;
  uint8_t* sA = sB + F_HALVES * nst * DG::STAGE;
  int* sX = reinterpret_cast<int*>(sA + slices * DG::SLICE);
  FBars* bars = reinterpret_cast<FBars*>(sX + F_HALVES * F_XRING * FN);

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);  // known to be uniform
  const int lane = threadIdx.x & 31;
  const int N = p.N, mtiles = (N + BM - 1) / BM;
  const int grp = blockIdx.x % groups, m0 = grp * slices;
  const int ms = mtiles - m0 < slices ? mtiles - m0 : slices;  // this CTA's slices
  const int64_t ntiles = (p.ncells + FN - 1) / FN;
  // warps 0-15 epilogue (half = warp / 8), 16-21 producers and 22-23 MMA (half = warp & 1)
  const int half = warp < F_PWARP0 ? warp / F_EPI : warp & 1;
  const int64_t t0 = (int64_t)(blockIdx.x / groups) * F_HALVES + half;  // this half's tiles: t0, t0 + tstep, ..
  const int64_t tstep = (int64_t)((gridDim.x - grp + groups - 1) / groups) * F_HALVES;

  if (threadIdx.x == 0) {
    for (int h = 0; h < F_HALVES; ++h) {
      for (int s = 0; s < F_STAGES; ++s) {
        mbar_init(smem_u32(&bars->full[h][s]), FN);
        mbar_init(smem_u32(&bars->empty[h][s]), 1);
      }
      mbar_init(smem_u32(&bars->tfull[h]), 1);
      mbar_init(smem_u32(&bars->tempty[h]), F_EPI);
      mbar_init(smem_u32(&bars->done[h]), 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == F_WARPS - 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tmem_base)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  {
    const uint4* src = reinterpret_cast<const uint4*>(p.digits + (size_t)m0 * DG::SLICE);
    uint4* dst = reinterpret_cast<uint4*>(sA);
    for (int i = threadIdx.x; i < ms * (DG::SLICE / 16); i += F_THREADS) dst[i] = __ldg(src + i);
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base + half * F_COLS;
  sB += half * nst * DG::STAGE;
  sX += half * F_XRING * FN;
  const uint32_t full = smem_u32(bars->full[half]), empty = smem_u32(bars->empty[half]);
  const uint32_t tfull = smem_u32(&bars->tfull[half]), tempty = smem_u32(&bars->tempty[half]);

  if (warp >= F_PWARP0 && warp < F_MWARP0) {
    // ---------------- producers: a tile per warp, a cell per thread ----------------
    int64_t i = (warp - F_PWARP0) >> 1;  // local tile number
    for (int64_t t = t0 + i * tstep; t < ntiles; t += F_PROD * tstep, i += F_PROD) {
      const int st = (int)(i % nst);
      const int64_t e = t * FN + lane;
      double G[K];
      int flag = 0;  // 0 digits, 1 skip, 2 plain
      if (e < p.ncells) {
        if (!factors64<FORM, D, true>(p, e, G)) {
          atomicOr(p.err, ERR_INDEX);
          flag = 1;
        }
      } else {
        flag = 1;
      }
      int X = 0;  // largest biased exponent of the scaled factors, in place (<< 20)
      if (!flag) {
        bool wild = false;
        uint32_t some = 0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          some |= (uint32_t)__double2hiint(G[k]) << 1 | (uint32_t)__double2loint(G[k]);
          const int ef = __double2hiint(G[k]) & 0x7FF00000;
          wild = wild || ef == 0x7FF00000;
          if (ef != 0) X = max(X, ef + p.tk20[term_of<FORM, D>(k)]);
        }
        wild = wild || (some != 0 && (X < (123 << 20) || X > (1923 << 20)));
        if (wild) flag = 2;
      }
      if (flag) {
#pragma unroll
        for (int k = 0; k < K; ++k) G[k] = 0.0;
      }
      // Parities tell only neighbouring phases apart. The warps are at most 2 tiles apart and there are 2
      // stages or more, so the stage's use before this one is the oldest whose tile may still be missing:
      // once it is full, its release is the phase that the second wait can mean.
      const uint32_t use = (uint32_t)(i / nst);
      if (use > 0 && !mbar_wait(full + 8 * st, (use - 1) & 1u, p.err)) break;
      if (!mbar_wait(empty + 8 * st, (use & 1u) ^ 1u, p.err)) break;
      uint8_t* dst = sB + st * DG::STAGE + lane * 16;
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        uint64_t U[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int k = 8 * c + j;
          U[j] = k < K ? fixed_point<DG::bias(), DG::FB>(G[k < K ? k : 0], X, p.tk20[term_of<FORM, D>(k < K ? k : 0)])
                       : DG::bias();
        }
        if (c == KC - 1) store_digits<B, ND, FN * 16, true>(dst + c * (ND * FN * 16), U);
        else store_digits<B, ND, FN * 16, false>(dst + c * (ND * FN * 16), U);
      }
      sX[(i % F_XRING) * FN + lane] = flag == 1 ? CELL_SKIP : flag == 2 ? CELL_PLAIN : X - (1022 << 20);
      fence_proxy_async();
      mbar_arrive(full + 8 * st);
    }
  } else if (warp >= F_MWARP0) {
    // ---------------- MMA issuer ----------------
    // Digit q of T against the cells' digits 0 .. ND-1-q at once: their 32-row blocks follow one another as
    // the orders' columns do, so one MMA of N = 32 (ND - q) adds to the orders q .. ND-1. An MMA takes 45 cycles
    // at N <= 64 and N / 2 from 128 on, its issue as long or longer, so few wide ones matter (advection-
    // diffusion: 24 a slice of 128 entries where an MMA per pair of digits and two K chunks took 92).
    if (lane == 0) {
      const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB);
      uint32_t slice = 0;
      int64_t i = 0;
      bool ok = true;
      for (int64_t t = t0; t < ntiles && ok; t += tstep, ++i) {
        const int s = (int)(i % nst);
        if (!mbar_wait(full + 8 * s, (uint32_t)((i / nst) & 1), p.err)) break;
        tc_fence_after();
        for (int m = 0; m < ms; ++m, ++slice) {
          if (!mbar_wait(tempty, (slice & 1u) ^ 1u, p.err)) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < KC; c += 2) {
            // the last chunk of an odd number: the other half of the K step is the table's zero chunk, against
            // which the cells' side may read any finite halves, here the table's
            const bool odd = c == KC - 1;
            const uint32_t bc = b0 + (uint32_t)(s * DG::STAGE + c * (ND * FN * 16));
            const uint64_t bd = f_desc(bc, odd ? a0 - bc : ND * FN * 16);
#pragma unroll
            for (int q = 0; q < ND; ++q) {
              const uint32_t chunk = (uint32_t)(q * KC + c);
              const uint64_t ad = f_desc(a0 + (uint32_t)(m * DG::SLICE) + chunk * (BM * 16),
                                         (odd ? (uint32_t)(ND * KC) - chunk : 1u) * (BM * 16));
              mma<false>(tmem + q * FN, ad, bd, make_idesc(0, BM, (ND - q) * FN), c | q ? 1u : 0u);
            }
          }
          tc_commit(tfull);
        }
        tc_commit(empty + 8 * s);
      }
      tc_commit(smem_u32(&bars->done[half]));
      mbar_wait(smem_u32(&bars->done[half]), 0, p.err);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue: orders combined in 64-bit integers, one rounding to double ----------------
    const int q = warp & 3, sub = (warp >> 2) & 1;  // TMEM lane quadrant; which cells of the tile
    const uint32_t tcol = tmem + ((uint32_t)(q * 32) << 16) + sub * FC;
    uint32_t slice = 0;
    bool ok = true;
    // the accumulators of orders d and d - 1 (r0, r1), of the latter alone with both = false
    auto load = [&](int d, uint32_t (&r0)[FC], uint32_t (&r1)[FC], bool both) {
      if (both) tmem_ld16(tcol + d * FN, r0);
      tmem_ld16(tcol + (d - 1) * FN, r1);
      tmem_wait_ld();
    };
    const uint32_t pB = opaque(1u << B), pB4 = opaque(1u << (B + 4)), p4 = opaque(16u), p18 = opaque(1u << 18),
                   p20 = opaque(1u << 20), p22 = opaque(1u << 22);
    const int npad = (N + 3) & ~3;
    int64_t i = 0;
    for (int64_t t = t0; t < ntiles && ok; t += tstep, ++i) {
      const int64_t cbase = t * FN + sub * FC;
      for (int m = 0; m < ms; ++m, ++slice) {
        const int o = (m0 + m) * BM + q * 32 + lane;
        // S = sum_d v_d 2^(B (1-d)) 2^36 over the orders d, from the accumulators' bits r_d = MAGIC + v_d. All
        // the constants of MAGIC are subtracted at once, as the high word of the first addend, HC: the
        // products keep them unsigned without a carry out, and their low words cancel (b = 9: order 3's
        // constant is 2^13 less; b = 8: by the constant added to the first term).
        constexpr uint32_t KP = MAGIC * ((1u << B) + 1u);  // constant of a pair of orders
        constexpr uint32_t C0 = MAGIC * ((1u << (B + 4)) + 16u);
        constexpr uint32_t HC = 0u - (B == 9 ? KP >> 14 : 9u + (KP >> 12)) - C0;
        uint32_t lo[FC], hi[FC];
        {
          uint32_t r0[FC], r1[FC];
          if (!mbar_wait(tfull, slice & 1u, p.err)) { ok = false; break; }
          __syncwarp();
          tc_fence_after();
          load(7, r0, r1, B == 8);  // orders 7 (b = 8, without the constant) and 6
#pragma unroll
          for (int j = 0; j < FC; ++j)
            lo[j] = B == 9 ? r1[j] >> 9
                           : (r1[j] >> 4) + (__float_as_uint(__uint_as_float(r0[j]) + 25165824.0f) >> 11) +
                                 (0x4C000000u - (MAGIC >> 4) - (0x4BC00000u >> 11));
          load(5, r0, r1, true);
#pragma unroll
          for (int j = 0; j < FC; ++j) {
            const uint32_t c = mad_lo(r1[j], pB, r0[j]);
            if constexpr (B == 9) {
              lo[j] = c + lo[j] + (0x80000000u - KP - (MAGIC >> 9));
            } else {
              const uint64_t S = mad_wide(c, p4, (uint64_t)HC << 32 | lo[j]);
              lo[j] = (uint32_t)S;
              hi[j] = (uint32_t)(S >> 32);
            }
          }
          load(3, r0, r1, true);
#pragma unroll
          for (int j = 0; j < FC; ++j) {
            const uint64_t S =
                mad_wide(mad_lo(r1[j], pB, r0[j]), B == 9 ? p18 : p20, (uint64_t)(B == 9 ? HC : hi[j]) << 32 | lo[j]);
            lo[j] = (uint32_t)S;
            hi[j] = (uint32_t)(S >> 32);
          }
        }
        // global assembly: the entries' positions, requested ahead of their use
        uint32_t pos[CSR ? FC : 1];
        if constexpr (CSR) {
          const int bw = npad - (o & ~31) < 32 ? npad - (o & ~31) : 32;  // width of this 32-entry map block
          const uint32_t* mp = p.map + 32 * ((t * FN >> 5) * (int64_t)npad + (o & ~31)) + sub * FC * bw + (o & 31);
#pragma unroll
          for (int j = 0; j < FC; ++j) pos[j] = o < N && cbase + j < p.ncells ? __ldg(mp + j * bw) : 0xffffffffu;
        }
        // orders 1 and 0: the high word alone
        {
          uint32_t r0[FC], r1[FC];
          load(1, r0, r1, true);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty);
#pragma unroll
          for (int j = 0; j < FC; ++j) hi[j] = mad_lo(r1[j], pB4, mad_lo(r0[j], p4, hi[j]));
        }
        if ((m0 + m) * BM + q * 32 >= N) continue;  // warp-uniform
        const int* xs = sX + (i % F_XRING) * FN + sub * FC;
        const bool special = __any_sync(0xffffffffu, xs[lane & (FC - 1)] <= CELL_PLAIN);
        const int y20 = o < N ? __ldg(p.yexp20 + o) : 0;
        bool rest = o < N;  // entries left for the general form
        if (!special && rest) {  // whole tiles of ordinary cells
          double* out = static_cast<double*>(p.out) + (CSR ? 0 : cbase * p.ostride + o);
          const int64_t stride = p.ostride;
          int least = 0;  // negative: some entry's high word is 0 or -1
          // eight at a time: their exponents loaded before any store (which the compiler must take for one to
          // the same memory), so that eight chains of dependent instructions run side by side
#pragma unroll
          for (int j0 = 0; j0 < FC; j0 += 8) {
            double v[8];
            int x[8], bit[8];
            *reinterpret_cast<int4*>(x) = *reinterpret_cast<const int4*>(xs + j0);
            *reinterpret_cast<int4*>(x + 4) = *reinterpret_cast<const int4*>(xs + j0 + 4);
#pragma unroll
            for (int j = 0; j < 8; ++j)
              v[j] = from_fixed(hi[j0 + j], lo[j0 + j], (uint32_t)(x[j] + y20), p22, p20, bit[j]);
            if constexpr (CSR) {
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                if (bit[j] < 0) v[j] = from_fixed_any(hi[j0 + j], lo[j0 + j], (uint32_t)(x[j] + y20));
                if (pos[j0 + j] < (uint64_t)p.nnz) atomicAdd(out + pos[j0 + j], v[j]);
                else atomicOr(p.err, ERR_INDEX);
              }
            } else {
#pragma unroll
              for (int j = 0; j < 8; j += 2) least |= bit[j] | bit[j + 1];
#pragma unroll
              for (int j = 0; j < 8; ++j) __stcs(out + (j0 + j) * stride, v[j]);
            }
          }
          rest = least < 0;
        }
        // a ragged tile, unusual cells, or an entry below 2^-24 of its cell's scale
        if (rest)
#pragma unroll
        for (int j = 0; j < FC; ++j) {
          const int64_t cell = cbase + j;
          const int x20 = xs[j];
          if (x20 == CELL_SKIP) continue;
          const double v =
              x20 == CELL_PLAIN ? plain_entry<FORM, D>(p, cell, o) : from_fixed_any(hi[j], lo[j], (uint32_t)(x20 + y20));
          if constexpr (CSR) {
            if (pos[j] < (uint64_t)p.nnz) atomicAdd(static_cast<double*>(p.out) + pos[j], v);
            else atomicOr(p.err, ERR_INDEX);
          } else {
            __stcs(static_cast<double*>(p.out) + cell * p.ostride + o, v);
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == F_WARPS - 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(bars->tmem_base), "r"(TMEM_COLS)
                 : "memory");
  }
}

constexpr int F_SMEM_LIMIT = 227 * 1024;
constexpr int F_FIXED = F_HALVES * F_XRING * FN * 4 + (int)sizeof(FBars) + 64;

template <int FORM, int D>
int fit_slices(int mtiles) {
  using DG = Digits<FORM, D>;
  const int fit = (F_SMEM_LIMIT - F_FIXED - F_HALVES * 2 * DG::STAGE) / DG::SLICE;
  if (fit >= mtiles) return mtiles;
  const int groups = (mtiles + fit - 1) / fit;  // even shares
  return (mtiles + groups - 1) / groups;
}

template <int FORM, int D>
cudaError_t launch_digits(const Fp64Params& p, int num_sms, cudaStream_t s) {
  using DG = Digits<FORM, D>;
  const int mtiles = (p.N + BM - 1) / BM, slices = fit_slices<FORM, D>(mtiles);
  const int groups = (mtiles + slices - 1) / slices;
  int nst = F_STAGES;
  while (slices * DG::SLICE + F_HALVES * nst * DG::STAGE + F_FIXED > F_SMEM_LIMIT) --nst;
  int smem = slices * DG::SLICE + F_HALVES * nst * DG::STAGE + F_FIXED;
  if (smem < 120 * 1024) smem = 120 * 1024;  // one CTA (one owner of all TMEM columns) per SM
  const int64_t ntiles = (p.ncells + FN - 1) / FN;
  const int grid = (int)std::min<int64_t>((ntiles + F_HALVES - 1) / F_HALVES * groups, num_sms);
  auto kern = p.map ? k_assemble_fp64_tc<FORM, D, true> : k_assemble_fp64_tc<FORM, D, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, F_THREADS, smem, s>>>(p, slices, groups, nst);
  return cudaGetLastError();
}

template <int FORM, int D>
void image_of(int degree, int cell, std::vector<uint8_t>& img, std::vector<int32_t>& y20, int32_t (&tk20)[2]) {
  using DG = Digits<FORM, D>;
  const int ns = nnodes(cell, degree), N = ns * ns, mtiles = (N + BM - 1) / BM;
  std::vector<double> T;
  reference_tensor(FORM, degree, cell, T);
  double top[2] = {0.0, 0.0};  // largest entry of each kind of term
  for (int k = 0; k < DG::K; ++k)
    for (int o = 0; o < N; ++o)
      top[term_of<FORM, D>(k)] = std::max(top[term_of<FORM, D>(k)], std::fabs(T[(size_t)k * N + o]));
  int tk[2];
  for (int j = 0; j < 2; ++j) {
    tk[j] = 0;
    if (top[j] > 0) std::frexp(top[j], &tk[j]);
    tk20[j] = tk[j] * (1 << 20);
  }
  img.assign((size_t)mtiles * DG::SLICE, 0);
  y20.assign(N, 0);
  for (int o = 0; o < N; ++o) {
    double big = 0.0;
    for (int k = 0; k < DG::K; ++k)
      big = std::max(big, std::fabs(std::ldexp(T[(size_t)k * N + o], -tk[term_of<FORM, D>(k)])));
    int y = 0;
    if (big > 0) std::frexp(big, &y);
    // S counts 2^-59 of 2^(x + y): order 1 weighs 2^36 in S and 2^-23 in the result (b = 9: leading digits
    // 2^-7 each, one order 2^-9), or 2^36 and 2^-20 (b = 8: 2^-6 each and 2^-8)
    y20[o] = (y - (DG::B == 9 ? 59 : 56) + 1054) * (1 << 20);
    uint8_t* slice = img.data() + (size_t)(o / BM) * DG::SLICE + (size_t)(o % BM) * 16;
    for (int q = 0; q < DG::ND; ++q) {
      const int block = q * DG::KC;  // digit q counts from the leading one
      for (int k = 0; k < DG::K; ++k) {
        const double f = std::nearbyint(std::ldexp(T[(size_t)k * N + o], DG::FB - tk[term_of<FORM, D>(k)] - y));
        const uint64_t U = (uint64_t)(int64_t)f + DG::bias();
        uint64_t u = U >> (DG::B * (DG::ND - 1 - q));
        if (q) u &= (1u << DG::B) - 1u;
        const uint16_t h = half_of_int((int)u - (1 << (DG::B - 1)));
        std::memcpy(slice + (size_t)(block + k / 8) * BM * 16 + (k % 8) * 2, &h, 2);
      }
      // the constant's other factor, 3072 (3070 in order 3 of the 9-bit digits, which takes 2^13 off the
      // constant; none in order 7 of the 8-bit digits)
      const uint16_t h = half_of_int(DG::B == 8 ? (q == 7 ? 0 : 3072) : q == 3 ? 3070 : 3072);
      std::memcpy(slice + (size_t)(block + DG::KC - 1) * BM * 16 + 14, &h, 2);
    }
  }
}

}  // namespace

// Where the digit contraction runs instead of the plain kernel: where it is the faster one at every count
// of cells, from 300 (both launch-bound, 8-20 us against 11-2300 us) to 196,608 (53-1100 us against
// 84-16,900 us). Left to the plain kernel are P1 triangles (9 entries: Helmholtz 32 against 47 us) and the
// mass matrices of up to 6 nodes (one multiplication an entry: P2 triangles at 300 cells 5 against 9 us).
int fp64_tc_use(int form, int degree, int cell) {
  const int ns = nnodes(cell, degree);
  if (form == FORM_MASS) return ns >= 10;
  return (form == FORM_HELMHOLTZ || form == FORM_ADVDIFF) && ns >= 4;
}

void build_fp64_image(int form, int degree, int cell, std::vector<uint8_t>& img, std::vector<int32_t>& y20,
                      int32_t (&tk20)[2]) {
  const bool tri = cell == CELL_TRI;
  if (form == FORM_MASS) {
    if (tri) image_of<FORM_MASS, 2>(degree, cell, img, y20, tk20);
    else image_of<FORM_MASS, 3>(degree, cell, img, y20, tk20);
  } else if (form == FORM_HELMHOLTZ) {
    if (tri) image_of<FORM_HELMHOLTZ, 2>(degree, cell, img, y20, tk20);
    else image_of<FORM_HELMHOLTZ, 3>(degree, cell, img, y20, tk20);
  } else {
    if (tri) image_of<FORM_ADVDIFF, 2>(degree, cell, img, y20, tk20);
    else image_of<FORM_ADVDIFF, 3>(degree, cell, img, y20, tk20);
  }
}

int launch_fp64_tc(int form, int cell, const Fp64Params& p, int num_sms, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool tri = cell == CELL_TRI;
  if (form == FORM_MASS)
    return (int)(tri ? launch_digits<FORM_MASS, 2>(p, num_sms, s) : launch_digits<FORM_MASS, 3>(p, num_sms, s));
  if (form == FORM_HELMHOLTZ)
    return (int)(tri ? launch_digits<FORM_HELMHOLTZ, 2>(p, num_sms, s) : launch_digits<FORM_HELMHOLTZ, 3>(p, num_sms, s));
  return (int)(tri ? launch_digits<FORM_ADVDIFF, 2>(p, num_sms, s) : launch_digits<FORM_ADVDIFF, 3>(p, num_sms, s));
}

}  // namespace coffee
