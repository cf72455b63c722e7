// FP64 local and global assembly on the tensor cores: A_e[o] = sum_k G_e[k] T[k][o] with the
// contraction done exactly, in integers, by tcgen05 f16 MMAs. (Matrix products from slices whose products are exact:
// Ozaki, Ogita, Oishi and Rump, Numerical Algorithms 59 (2012), 95-118.)
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
// 2^-56 of max_k |G_k| max_k |T_k|, where K rounded FMAs stood before.
//
// That is no more than the FMAs' error only where some term G_k T_k is of that order. So a cell has a mask of its
// factors above 1/8 of its largest, an entry one of its table column above 1/8 of the largest there, and where
// the two have no bit in common (an entry of stretched or right-angled cells whose large factors meet zeros of T)
// the producers, which have the factors of a cell in each thread, take the sum in FP64 and store it, and the epilogue
// leaves that entry out (weak_entries). Elsewhere sum_k |G_k T_k| is at least 2^-8 of the product of the largest. The
// cost goes with what it does: 0.4 % of the entries of perturbed P3 tetrahedra, a fifth to a half of them on thin
// layers, all entries of cells whose factors are not finite or outside 2^+-900, which have no digits.
// Error of an entry against quadruple precision relative to its own sum_k |G_k T_k|, rms in units of 2^-53, this kernel /
// plain: Helmholtz P3 tetrahedra perturbed 0.90 / 0.94, right-angled 0.24 / 0.34; advection-diffusion P2 perturbed 1.32 /
// 1.38, right-angled 0.43 / 0.62, with eps = 1e-6 0.56 / 0.59; P3 triangles 0.51 / 0.71, in layers of 1/1000 0.72 / 0.88. No
// rms is larger; the largest errors are the same (the factors' own) or within 1.2 times, but for triangles in layers,
// 11 / 5.6. Without the masks the largest were 1e4 (right-angled) to 1e8 (layers).
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
// moved to the multiplier pipe, see mad_lo), and the latencies between its phases; for advection-diffusion the
// producers. 196,608 perturbed tetrahedra (thin layers), this kernel / plain: Helmholtz P2 80 (193) / 302 us, P3 155
// (477) / 1140 us, 0.6 of the copy bandwidth, P4 381 (1230) / 3480 us; advection-diffusion P1 175 (280) / 276, P2 183
// (559) / 1450 us, P3 0.76 (2.31) / 5.41 ms. Steps on the way (Helmholtz P3): one
// pipeline with 21 warps 479 us; 16 warps of 128 registers 324; multiplications for shifts 311; two
// pipelines 242; 16 cells per epilogue warp, four epilogue warps a scheduler, 169; one wide MMA per digit of T
// instead of one per order and K step 158 (advection-diffusion P2 168 -> 123). The masks and weak_entries took
// advection-diffusion P2 from 123 to 183 us and Helmholtz P2 from 59 to 80.
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <map>
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
constexpr int CELL_SKIP = INT32_MIN;
constexpr int F_WEAK = 3;              // a factor or table entry counts as large above 2^-3 of the largest
constexpr uint32_t MAGIC = 0x4B400000u;  // 1.5 * 2^23 as a float

struct alignas(8) FBars {
  uint64_t full[F_HALVES][F_STAGES], empty[F_HALVES][F_STAGES], tfull[F_HALVES], tempty[F_HALVES], done[F_HALVES],
      stored[F_HALVES][F_PROD];
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
  static constexpr int KP = K < 8 ? 8 : K < 16 ? 16 : 40;  // words of an entry's row for weak_entries: T[k], zeros, the entry last
  COFFEE_HD static constexpr uint64_t bias() {
    uint64_t s = 0;
    for (int p = 0; p < ND; ++p) s += 1ull << (B - 1 + B * p);
    return s;
  }
};

// Whether the epilogue leaves weak_entries' entries out, so that these need not wait for it: global assembly, which adds,
// and advection-diffusion on tetrahedra, whose producers the wait holds up (P3 809 us, 990 with it; on triangles it
// is the test per store that costs: P4 135 us, 115 without).
template <int FORM, int D, bool CSR>
__device__ constexpr bool leaves() { return CSR || (FORM == FORM_ADVDIFF && D == 3); }

// The entries of the warp's 32 cells (one per lane, factors G; live: to be stored at all) that have no large term, or all of
// cells without digits (big = 0): their sums in FP64 over all terms, as the plain kernel takes them. Element matrices:
// stored over what the epilogue wrote, after it has stored the tile (phase n of the barrier `stored`). The entries come
// in classes of one mask of large table entries, whose rows of T lie one after the other, the entry's number last.
// Few cells fail a class (perturbed tetrahedra: 40 pairs of a cell and an entry in a tile), so pairs are queued and summed
// 32 at a time, a pair per lane with the factors from their cell's lane: class by class for all lanes, advection-diffusion
// P2 on 196,608 tetrahedra took 415 us, now 183. Called by whole warps, and every lane takes part in every
// exchange; false on expiry.
template <int FORM, int D, bool CSR>
__device__ __forceinline__ bool weak_entries(const Fp64Params& p, int64_t e0, bool live, uint32_t big,
                                             const Factors<FORM, D>& G, int grp, uint32_t* queue,
                                             uint32_t stored, uint32_t n) {
  using DG = Digits<FORM, D>;
  constexpr int K = DG::K, KP = DG::KP;
  constexpr uint32_t FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, npad = (p.N + 3) & ~3;
  const int4* classes = reinterpret_cast<const int4*>(p.classes);
  const int2 range = __ldg(reinterpret_cast<const int2*>(p.groups) + grp);
  const uint32_t common = __reduce_and_sync(FULL, live ? big : FULL);
  int queued = 0;
  bool waited = leaves<FORM, D, CSR>();
  auto flush = [&](int count) {  // the queue's first pairs
    __syncwarp();
    const uint32_t q = queue[lane < count ? lane : 0];
    const int cell = (int)(q & 31u);
    const double2* row = reinterpret_cast<const double2*>(static_cast<const double*>(p.weak) + (int64_t)(q >> 5) * KP);
    const int o = (int)__double_as_longlong(__ldg(row + KP / 2 - 1).y);
    double T[KP - 1];
#pragma unroll
    for (int k = 0; k < K; k += 2) {
      const double2 w = __ldg(row + k / 2);
      T[k] = w.x;
      if (k + 1 < K) T[k + 1] = w.y;
    }
    auto of = [&](int x) { return __shfl_sync(FULL, G.f[x], cell); };
    double acc = 0.0;
    if constexpr (FORM == FORM_ADVDIFF) {
      constexpr int NV = D + 1, P = D * (D + 1) / 2;
      double H[P];
#pragma unroll
      for (int x = 0; x < P; ++x) H[x] = of(x);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        double s = 0.0;
#pragma unroll
        for (int x = 0; x < P; ++x) s = fma(H[x], T[v * P + x], s);
        acc = fma(of(P + v), s, acc);
      }
#pragma unroll
      for (int x = 0; x < NV * D; ++x) acc = fma(of(P + NV + x), T[NV * P + x], acc);
    } else {
#pragma unroll
      for (int k = 0; k < K; ++k) acc = fma(of(k), T[k], acc);
    }
    if (lane < count) {
      const int64_t e = e0 + cell;
      if constexpr (CSR) {
        const uint32_t pos = __ldg(p.map + csr_map_index(e, o, npad));
        if (pos < (uint64_t)p.nnz) atomicAdd(static_cast<double*>(p.out) + pos, acc);
        else atomicOr(p.err, ERR_INDEX);
      } else {
        __stcs(static_cast<double*>(p.out) + e * p.ostride + o, acc);
      }
    }
    __syncwarp();
  };
  // (one place that sums: inlined twice, advection-diffusion's code waited for instructions, P2 205 us)
  int4 cl = make_int4(0, 0, 0, 0);   // 32 classes on the lanes: mask, first row, last row + 1
  uint32_t hits = 0, fails = 0;      // of them, those that not every cell has a large factor of; the cells that fail the class
  int c0 = range.x, i = 0, last = 0;  // next classes, next row of the class
  for (;;) {
    while (queued < 32) {
      if (i == last) {
        for (; hits == 0u && c0 < range.y; c0 += 32) {
          cl = c0 + lane < range.y ? __ldg(classes + c0 + lane) : make_int4(-1, 0, 0, 0);
          hits = __ballot_sync(FULL, (common & (uint32_t)cl.x) == 0u && cl.y < cl.z);
        }
        if (hits == 0u) break;
        const int src = __ffs(hits) - 1;
        hits &= hits - 1;
        const uint32_t mask = (uint32_t)__shfl_sync(FULL, cl.x, src);
        i = __shfl_sync(FULL, cl.y, src);
        last = __shfl_sync(FULL, cl.z, src);
        fails = __ballot_sync(FULL, live && (big & mask) == 0u);
        if (fails == 0u) i = last;
        continue;
      }
      if (fails >> lane & 1u) queue[queued + __popc(fails & ((1u << lane) - 1u))] = (uint32_t)i << 5 | (uint32_t)lane;
      queued += __popc(fails);
      ++i;
    }
    if (queued == 0) return true;
    if (!waited) {
      if (!__all_sync(FULL, mbar_wait(stored, n & 1u, p.err))) return false;
      waited = true;
    }
    const int count = queued < 32 ? queued : 32;
    flush(count);
    queued -= count;
    const uint32_t rest = queue[32 + lane];
    __syncwarp();
    if (lane < queued) queue[lane] = rest;
    __syncwarp();
  }
}

// The largest biased exponent X of a cell's scaled factors, in place (<< 20; 0: all are zero), and the mask `big` of those
// (of the first 32) that are at least 2^-3 of 2^(X - 1023); false: the cell has no digits, big = 0. Advection-diffusion
// takes the largest product eps H from the largest factors and the others' sizes from the sums of their logarithms,
// as the high words give these within 0.09 and never too large: the FP64 pipe, which the products would take a
// second and third time, is what bounds its producers.
template <int FORM, int D>
__device__ __forceinline__ bool scale_of(const Factors<FORM, D>& G, const int32_t (&tk20)[2], int& X, uint32_t& big) {
  constexpr int NV = D + 1, P = D * (D + 1) / 2, K = FormK<FORM, D>::value;
  auto high = [](double x) { return __double2hiint(x) & 0x7FFFFFFF; };
  auto bits = [](double x) -> uint64_t { return (uint64_t)__double_as_longlong(x) & ~(1ull << 63); };
  constexpr int E = 0x7FF00000;
  bool wild = false;
  uint64_t some = 0;
  auto take = [&](double g, int t20) {
    some |= bits(g);
    const int ef = high(g) & E;
    wild = wild || ef == E;
    if (ef != 0) X = max(X, ef + t20);
  };
  X = 0;
  if constexpr (FORM == FORM_ADVDIFF) {
    uint64_t h = 0, c = 0;
#pragma unroll
    for (int x = 0; x < P; ++x) h = max(h, bits(G.f[x]));
#pragma unroll
    for (int x = 0; x < NV; ++x) c = max(c, bits(G.f[P + x]));
    wild = h >> 52 == 0x7FFu || c >> 52 == 0x7FFu;
    take(__longlong_as_double((int64_t)h) * __longlong_as_double((int64_t)c), tk20[0]);
#pragma unroll
    for (int x = 0; x < NV * D; ++x) take(G.f[P + NV + x], tk20[1]);
  } else {
#pragma unroll
    for (int k = 0; k < K; ++k) take(G.f[k], tk20[term_of<FORM, D>(k)]);
  }
  wild = wild || (some != 0 && (X < (123 << 20) || X > (1923 << 20)));
  big = some != 0 || wild ? 0u : ~0u;
  if (some != 0 && !wild) {
    const int least = X - (F_WEAK << 20);
#pragma unroll
    for (int k = 0; k < (K < 32 ? K : 32); ++k) {
      bool b;
      if (FORM == FORM_ADVDIFF && k < NV * P) {
        const int x = high(G.f[k % P < Factors<FORM, D>::COUNT ? k % P : 0]);
        const int y = high(G.f[P + k / P < Factors<FORM, D>::COUNT ? P + k / P : 0]);
        b = x >= 1 << 20 && y >= 1 << 20 && x + y - (1023 << 20) + tk20[0] >= least;
      } else {
        const int x = high(G.at(k));
        b = x >= 1 << 20 && x + tk20[term_of<FORM, D>(k)] >= least;
      }
      if (b) big |= 1u << k;
    }
  }
  return !wild;
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
  uint32_t* sM = reinterpret_cast<uint32_t*>(sX + F_HALVES * F_XRING * FN);
  uint32_t* sQ = sM + F_HALVES * F_XRING * FN;  // queues of weak_entries, 64 words a producer warp
  FBars* bars = reinterpret_cast<FBars*>(sQ + F_HALVES * F_PROD * 64);

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
      for (int w = 0; w < F_PROD; ++w) mbar_init(smem_u32(&bars->stored[h][w]), F_EPI);
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
  sM += half * F_XRING * FN;
  const uint32_t full = smem_u32(bars->full[half]), empty = smem_u32(bars->empty[half]);
  const uint32_t tfull = smem_u32(&bars->tfull[half]), tempty = smem_u32(&bars->tempty[half]);

  if (warp >= F_PWARP0 && warp < F_MWARP0) {
    // ---------------- producers: a tile per warp, a cell per thread ----------------
    const int w = (warp - F_PWARP0) >> 1;
    const uint32_t stored = smem_u32(&bars->stored[half][w]);
    int64_t i = w;  // local tile number
    for (int64_t t = t0 + i * tstep; t < ntiles; t += F_PROD * tstep, i += F_PROD) {
      const int st = (int)(i % nst);
      const int64_t e = t * FN + lane;
      Factors<FORM, D> G;
      int flag = 0;  // 0 digits, 1 skip, 2 no digits
      if (e < p.ncells) {
        if (!factors64<FORM, D, true>(p, e, G)) {
          atomicOr(p.err, ERR_INDEX);
          flag = 1;
        }
      } else {
        flag = 1;
      }
      int X = 0;  // largest biased exponent of the scaled factors, in place (<< 20)
      uint32_t big = ~0u;  // the factors above 2^-3 of the largest, of the first 32
      if (!flag && !scale_of<FORM, D>(G, p.tk20, X, big)) flag = 2;
      if constexpr (FORM != FORM_MASS)
        if (flag == 2) factors64<FORM, D, false>(p, e, G);  // infinities and NaN as divisions give them
      // Parities tell only neighbouring phases apart. This warp's tile before, i - 3, was stored after tile i - 3 - nst had
      // been contracted, so with 3 stages or more (one per producer warp) the stage's use before the last, tile i - 2 nst,
      // is over: the first wait can only mean the last use, tile i - nst, and once that is full, the second its release.
      const uint32_t use = (uint32_t)(i / nst);
      const uint32_t n = (uint32_t)(i / F_PROD);  // of this warp's tiles
      bool ok = use == 0 || mbar_wait(full + 8 * st, (use - 1) & 1u, p.err);
      ok = ok && mbar_wait(empty + 8 * st, (use & 1u) ^ 1u, p.err);
      // the warp's tile before has been stored: while this one is not on its way, its phase cannot be over, so the
      // parity means the one before, and that of the wait in weak_entries this one
      if (!leaves<FORM, D, CSR>()) ok = ok && (n == 0 || mbar_wait(stored, (n - 1) & 1u, p.err));
      if (!__all_sync(0xffffffffu, ok)) break;
      uint8_t* dst = sB + st * DG::STAGE + lane * 16;
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        uint64_t U[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int k = 8 * c + j;
          U[j] = k < K ? fixed_point<DG::bias(), DG::FB>(flag ? 0.0 : G.at(k < K ? k : 0), X, p.tk20[term_of<FORM, D>(k < K ? k : 0)])
                       : DG::bias();
        }
        if (c == KC - 1) store_digits<B, ND, FN * 16, true>(dst + c * (ND * FN * 16), U);
        else store_digits<B, ND, FN * 16, false>(dst + c * (ND * FN * 16), U);
      }
      sX[(i % F_XRING) * FN + lane] = flag == 1 ? CELL_SKIP : X - (1022 << 20);
      sM[(i % F_XRING) * FN + lane] = big;
      fence_proxy_async();
      mbar_arrive(full + 8 * st);
      if (!weak_entries<FORM, D, CSR>(p, t * FN, flag != 1, big, G, grp, sQ + (half * F_PROD + w) * 64, stored, n)) break;
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
        const uint32_t* ms = sM + (i % F_XRING) * FN + sub * FC;
        constexpr bool LEAVES = leaves<FORM, D, CSR>();
        const uint32_t mo = LEAVES && o < N ? __ldg(p.emask + o) : 0u;
        const bool special = __any_sync(0xffffffffu, xs[lane & (FC - 1)] == CELL_SKIP);
        const int y20 = o < N ? __ldg(p.yexp20 + o) : 0;
        uint32_t rest = o < N ? 0xffffu : 0u;  // entries left for the general form, cell j at bit 15 - j
        if (!special && rest) {  // whole tiles
          double* out = static_cast<double*>(p.out) + (CSR ? 0 : cbase * p.ostride + o);
          const int64_t stride = p.ostride;
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
            uint32_t c[8];
            if constexpr (LEAVES) {
              *reinterpret_cast<uint4*>(c) = *reinterpret_cast<const uint4*>(ms + j0);
              *reinterpret_cast<uint4*>(c + 4) = *reinterpret_cast<const uint4*>(ms + j0 + 4);
            }
            if constexpr (CSR) {
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                if ((c[j] & mo) == 0u) continue;
                if (bit[j] < 0) v[j] = from_fixed_any(hi[j0 + j], lo[j0 + j], (uint32_t)(x[j] + y20));
                if (pos[j0 + j] < (uint64_t)p.nnz) atomicAdd(out + pos[j0 + j], v[j]);
                else atomicOr(p.err, ERR_INDEX);
              }
            } else {
#pragma unroll
              for (int j = 0; j < 8; ++j) rest = __funnelshift_l((uint32_t)bit[j], rest, 1);
#pragma unroll
              for (int j = 0; j < 8; ++j)
                if (!LEAVES || (c[j] & mo) != 0u) __stcs(out + (j0 + j) * stride, v[j]);
            }
          }
          rest = CSR ? 0u : rest & 0xffffu;
        }
        // a ragged tile, cells with a bad index, or an entry below 2^-24 of its cell's scale
        if (rest)
#pragma unroll
        for (int j = 0; j < FC; ++j) {
          const int x20 = xs[j];
          if (!(rest >> (FC - 1 - j) & 1u) || x20 == CELL_SKIP || (LEAVES && (ms[j] & mo) == 0u)) continue;
          const double v = from_fixed_any(hi[j], lo[j], (uint32_t)(x20 + y20));
          if constexpr (CSR) {
            if (pos[j] < (uint64_t)p.nnz) atomicAdd(static_cast<double*>(p.out) + pos[j], v);
            else atomicOr(p.err, ERR_INDEX);
          } else {
            __stcs(static_cast<double*>(p.out) + (cbase + j) * p.ostride + o, v);
          }
        }
      }
      __syncwarp();
      if (!leaves<FORM, D, CSR>() && lane == 0) mbar_arrive(smem_u32(&bars->stored[half][i % F_PROD]));
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
constexpr int F_FIXED = F_HALVES * F_XRING * FN * 8 + F_HALVES * F_PROD * 64 * 4 + (int)sizeof(FBars) + 64;

template <int FORM, int D>
int fit_slices(int mtiles) {
  using DG = Digits<FORM, D>;
  // a stage for every producer warp (see the waits there)
  static_assert(F_SMEM_LIMIT - F_FIXED - F_HALVES * F_PROD * DG::STAGE >= DG::SLICE && F_STAGES >= F_PROD, "stages");
  const int fit = (F_SMEM_LIMIT - F_FIXED - F_HALVES * F_PROD * DG::STAGE) / DG::SLICE;
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
void image_of(int degree, int cell, std::vector<uint8_t>& img, Fp64Image& h) {
  using DG = Digits<FORM, D>;
  std::vector<int32_t>& y20 = h.y20;
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
    h.tk20[j] = tk[j] * (1 << 20);
  }
  img.assign((size_t)mtiles * DG::SLICE, 0);
  y20.assign(N, 0);
  h.emask.assign(N, 0);
  std::map<uint32_t, std::vector<int>> by_mask;
  for (int o = 0; o < N; ++o) {
    double big = 0.0;
    for (int k = 0; k < DG::K; ++k)
      big = std::max(big, std::fabs(std::ldexp(T[(size_t)k * N + o], -tk[term_of<FORM, D>(k)])));
    int y = 0;
    if (big > 0) std::frexp(big, &y);
    for (int k = 0; k < DG::K && k < 32; ++k)
      if (std::fabs(std::ldexp(T[(size_t)k * N + o], -tk[term_of<FORM, D>(k)])) >= std::ldexp(big, -F_WEAK)) h.emask[o] |= 1u << k;
    by_mask[h.emask[o]].push_back(o);
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
        const uint16_t c = half_of_int((int)u - (1 << (DG::B - 1)));
        std::memcpy(slice + (size_t)(block + k / 8) * BM * 16 + (k % 8) * 2, &c, 2);
      }
      // the constant's other factor, 3072 (3070 in order 3 of the 9-bit digits, which takes 2^13 off the
      // constant; none in order 7 of the 8-bit digits)
      const uint16_t c = half_of_int(DG::B == 8 ? (q == 7 ? 0 : 3072) : q == 3 ? 3070 : 3072);
      std::memcpy(slice + (size_t)(block + DG::KC - 1) * BM * 16 + 14, &c, 2);
    }
  }
  // classes and rows, for each group of CTAs those of its entries
  const int slices = fit_slices<FORM, D>(mtiles);
  for (int m0 = 0; m0 < mtiles; m0 += slices) {
    h.groups.push_back((int32_t)(h.classes.size() / 4));
    for (const auto& m : by_mask) {
      const int32_t first = (int32_t)(h.weak.size() / DG::KP);
      for (int o : m.second) {
        if (o / BM < m0 || o / BM >= m0 + slices) continue;
        const int64_t number = o;
        const size_t at = h.weak.size();
        h.weak.resize(at + DG::KP, 0.0);
        for (int k = 0; k < DG::K; ++k) h.weak[at + k] = T[(size_t)k * N + o];
        std::memcpy(&h.weak[at + DG::KP - 1], &number, 8);
      }
      const int32_t last = (int32_t)(h.weak.size() / DG::KP);
      if (last > first)
        for (int32_t x : {(int32_t)m.first, first, last, 0}) h.classes.push_back(x);
    }
    h.groups.push_back((int32_t)(h.classes.size() / 4));
  }
}

}  // namespace

// Where the digit contraction runs instead of the plain kernel: where it is the faster one at every count of cells
// from 300 (both launch-bound, 8-20 us against 11-2300 us) and on perturbed meshes as on thin layers, or nearly so. us,
// 196,608 cells perturbed, layered / plain: advection-diffusion P1 tetrahedra 175, 280 / 276, P2 triangles 70, 123 / 223;
// Helmholtz P2 tetrahedra 80, 193 / 302, P4 triangles 87, 182 / 570. Left to the plain kernel are
// Helmholtz on fewer than 10 nodes (P2 triangles 70, 119 / 76, P1 tetrahedra 74, 107 / 86, P1 triangles 47 / 32) and the
// mass matrices of up to 6 nodes (one multiplication an entry: P2 triangles at 300 cells 5 against 9 us).
int fp64_tc_use(int form, int degree, int cell) {
  const int ns = nnodes(cell, degree);
  return form == FORM_MASS || form == FORM_HELMHOLTZ ? ns >= 10 : form == FORM_ADVDIFF && ns >= 4;
}

void build_fp64_image(int form, int degree, int cell, std::vector<uint8_t>& img, Fp64Image& h) {
  const bool tri = cell == CELL_TRI;
  if (form == FORM_MASS) {
    if (tri) image_of<FORM_MASS, 2>(degree, cell, img, h);
    else image_of<FORM_MASS, 3>(degree, cell, img, h);
  } else if (form == FORM_HELMHOLTZ) {
    if (tri) image_of<FORM_HELMHOLTZ, 2>(degree, cell, img, h);
    else image_of<FORM_HELMHOLTZ, 3>(degree, cell, img, h);
  } else {
    if (tri) image_of<FORM_ADVDIFF, 2>(degree, cell, img, h);
    else image_of<FORM_ADVDIFF, 3>(degree, cell, img, h);
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
