// tcgen05 local assembly of element matrices that do not start on 32-byte sectors (P4: rows of 225 and 1225 floats).
//
// With the entries on the TMEM lanes, k_assemble_tc's warps store 32 consecutive entries of a cell: 128 bytes that
// straddle five sectors when the row's offset is odd, two of them shared with stores of another slice or cell at
// another time, which L2 fills from DRAM (P4 tetrahedra, contiguous rows: 4.8 sectors a store, 71 MB of fills for
// 0.96 GB; 2.92 ms for 1,572,864 cells where rows padded to 128 bytes take 1.56).
// Here every warp store covers four whole sectors. The offset r of a row within its sector, in floats, depends
// only on the cell modulo G = 8 / gcd(stride, 8): the tile's cells are sorted by that class in the B operand, and
// each class is contracted by MMAs of its own against T^T shifted down by r, so that lane l of slice m holds entry
// 128 m + l - r. The shift is free: T^T's 16-byte rows (8 zero rows first) are contiguous for each 16-byte K
// chunk, so a slice may start at any row. Tiles of 256 cells keep a class's MMA 32 cells wide (G = 8): an MMA
// takes 45 cycles at any N up to 64, and tiles of 128 cells, twice the MMAs, were bound by them (293 us for 196,608
// cells). Two slices go through one hand-off (one took 222 us, and 246 with one set of epilogue warps). Each CTA
// has one contiguous range of cells, so that no wave of tiles is left partly empty. 196,608 P4 tetrahedra 363 -> 170 us
// (0.84 of the copy bandwidth), 1,572,864 2920 -> 1180 us (0.97); 2^21 P4 triangles 640 -> 320 us (0.89).
// Roles as in k_assemble_tc: warps 0-3 and 13-16 epilogue, 4-11 producers (a cell each, both groups on one
// tile), 12 MMA.
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cstdint>
#include "coffee_internal.h"
#include "tc_common.cuh"

namespace coffee {
namespace {

using namespace tc;

constexpr int HN = 256;                // cells per tile
constexpr int H_STAGES = 2;
constexpr int H_THREADS = 17 * 32;     // NTHREADS and a second set of epilogue warps, 13-16

template <int FORM, int D, int PREC>
__global__ void __launch_bounds__(H_THREADS, 1) k_assemble_tc_shift(const TcParams p, int64_t range) {
  using PT = PrecTraits<PREC>;
  using PS = Passes<PREC>;
  constexpr int KP = round_up(Form<FORM, D>::K, PT::tf32 ? 8 : 16);
  constexpr int KB = KP * (PT::tf32 ? 4 : 2), KSTEPS = KB / 32;  // bytes of an operand row, MMA K steps
  constexpr int TPARTS = PT::TPARTS, GPARTS = PT::GPARTS;
  constexpr int GPART = HN * KB;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const int N = p.N, mtiles = p.mtiles, rows = mtiles * BM + 8;  // rows of T^T
  const int a_part = rows * KB;
  uint8_t* sA = smem_raw;
  uint8_t* sB = sA + TPARTS * a_part;
  Barriers* bars = reinterpret_cast<Barriers*>(sB + H_STAGES * GPARTS * GPART);
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int classes = p.classes, cg = HN / classes, nslot = TMEM_COLS / (2 * cg);  // cells of a class, accumulator pairs
  const int off0 = (int)((reinterpret_cast<uintptr_t>(p.out) >> 2) & 7), step = (int)(p.ostride & 7);
  const int64_t first = blockIdx.x * range, end = first + range < p.ncells ? first + range : p.ncells;

  if (threadIdx.x == 0) {
    for (int s = 0; s < H_STAGES; ++s) {
      mbar_init(smem_u32(&bars->full[s]), HN);
      mbar_init(smem_u32(&bars->empty[s]), 1);
    }
    for (int r = 0; r < MAX_SLOTS; ++r) {
      mbar_init(smem_u32(&bars->tfull[r]), 1);
      mbar_init(smem_u32(&bars->tempty[r]), EPI_WARPS);
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
  {
    const uint4* src = reinterpret_cast<const uint4*>(p.image);
    uint4* dst = reinterpret_cast<uint4*>(sA);
    for (int i = threadIdx.x; i < TPARTS * a_part / 16; i += H_THREADS) dst[i] = __ldg(src + i);
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;

  if (warp >= PROD_WARP0 && warp < MMA_WARP) {
    // ---------------- producers ----------------
    const int c = (warp - PROD_WARP0) * 32 + lane;  // cell of the tile
    const int brow = (c & (classes - 1)) * cg + c / classes;
    CellIds<FORM, D> ids{}, nids{};
    if (first + c < end) load_ids<FORM, D>(p, first + c, nids);
    uint32_t i = 0;
    for (int64_t t = first; t < end; t += HN, ++i) {
      const int64_t e = t + c;
      ids = nids;
      if (e + HN < end) load_ids<FORM, D>(p, e + HN, nids);
      const uint32_t s = i % H_STAGES;
      if (!mbar_wait(smem_u32(&bars->empty[s]), ((i / H_STAGES) & 1u) ^ 1u, p.err)) break;
      float G[KP];
      bool bad = false;
      if (e < end) {
        cell_factors_ids<FORM, D, KP>(p, ids, G, bad);
        if (bad) atomicOr(p.err, ERR_INDEX);
      }
      if (e >= end || bad) {
#pragma unroll
        for (int k = 0; k < KP; ++k) G[k] = 0.f;
      }
      store_operand_row<PREC, KP>(sB + s * (GPARTS * GPART), GPART, brow, G, KB);
      fence_proxy_async();
      mbar_arrive(smem_u32(&bars->full[s]));
    }
  } else if (warp == MMA_WARP) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB);
      const uint32_t idesc = make_idesc(PT::tf32 ? 2 : 1, BM, cg);
      uint32_t rc = 0, i = 0;
      bool ok = true;
      for (int64_t t = first; t < end && ok; t += HN, ++i) {
        const uint32_t s = i % H_STAGES;
        if (!mbar_wait(smem_u32(&bars->full[s]), (i / H_STAGES) & 1u, p.err)) break;
        tc_fence_after();
        const int some = end - t < classes ? (int)(end - t) : classes;  // classes that have cells
        for (int cls = 0; cls < some && ok; ++cls) {
          const uint64_t bd = make_desc(b0 + s * (GPARTS * GPART) + (uint32_t)(cls * cg * KB), 8 * KB);
          const int r = (off0 + cls * step) & 7;
          for (int m0 = 0; m0 < mtiles; m0 += 2, ++rc) {
            const uint32_t slot = rc % nslot;
            if (!mbar_wait(smem_u32(&bars->tempty[slot]), ((rc / nslot) & 1u) ^ 1u, p.err)) { ok = false; break; }
            tc_fence_after();
            for (int m = m0; m < mtiles && m < m0 + 2; ++m) {
              const uint64_t ad = make_desc_k(a0 + (uint32_t)((m * BM + 8 - r) * 16), (uint32_t)rows * 16, 128);
              const uint32_t d = tmem + slot * 2 * cg + (m - m0) * cg;
#pragma unroll
              for (int ks = 0; ks < KSTEPS; ++ks)
#pragma unroll
                for (int x = 0; x < PS::N; ++x)  // descriptor addresses count 16 bytes
                  mma<PT::tf32>(d, ad + (uint32_t)((PS::t(x) * KB / 16 + 2 * ks) * rows),
                                bd + PS::g(x) * (GPART / 16) + ks * 16, idesc, (ks | x) ? 1u : 0u);
            }
            tc_commit(smem_u32(&bars->tfull[slot]));
          }
        }
        tc_commit(smem_u32(&bars->empty[s]));
      }
      tc_commit(smem_u32(&bars->done));
      mbar_wait(smem_u32(&bars->done), 0, p.err);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue ----------------
    const int q = warp & 3;  // TMEM lane quadrant
    const uint32_t set = warp > MMA_WARP;  // two sets on alternate accumulators (there is an even number of them)
    const int64_t cstep = classes * p.ostride;  // from a cell to the next of its class
    uint32_t rc = 0;
    bool ok = true;
    for (int64_t t = first; t < end && ok; t += HN) {
      const int rem = end - t < HN ? (int)(end - t) : HN;
      const int some = rem < classes ? rem : classes;
      for (int cls = 0; cls < some && ok; ++cls) {
        const int o0 = q * 32 + lane - ((off0 + cls * step) & 7);
        for (int m = 0; m < mtiles; m += 2, ++rc) {
          if ((rc & 1u) != set) continue;
          const uint32_t slot = rc % nslot;
          if (!mbar_wait(smem_u32(&bars->tfull[slot]), (rc / nslot) & 1u, p.err)) { ok = false; break; }
          __syncwarp();
          tc_fence_after();
          const int blocks = 2 * cg / 32;  // of 32 columns: the first slice's cells, then the second's
#pragma unroll 1
          for (int b = 0; b < blocks; ++b) {
            const int h = b * 32 >= cg, k = b * 32 - h * cg, o = (m + h) * BM + o0;
            uint32_t v[32];
            tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + slot * 2 * cg + b * 32, v);
            tmem_wait_ld();
            if (b == blocks - 1) {  // read in full: the accumulators go back before the last stores
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(smem_u32(&bars->tempty[slot]));
            }
            if (o >= 0 && o < N) {
              float* dst = p.out + (t + cls + k * classes) * p.ostride + o;
              if (cls + (k + 31) * classes < rem) {
#pragma unroll
                for (int j = 0; j < 32; ++j) __stcs(dst + j * cstep, __uint_as_float(v[j]));
              } else {
#pragma unroll
                for (int j = 0; j < 32; ++j)
                  if (cls + (k + j) * classes < rem) __stcs(dst + j * cstep, __uint_as_float(v[j]));
              }
            }
            __syncwarp();
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == MMA_WARP) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

int shift_smem(int mtiles, int kbytes, int precision) {
  return prec_tparts(precision) * (mtiles * BM + 8) * kbytes + H_STAGES * prec_gparts(precision) * HN * kbytes +
         (int)sizeof(Barriers) + 64;
}

template <int FORM, int D, int PREC>
cudaError_t launch_shift_typed(const TcParams& p, int num_sms, cudaStream_t s, int smem) {
  // contiguous ranges of equal length, a multiple of the 32 cells that keep the classes in place
  const int64_t range = ((p.ncells + num_sms - 1) / num_sms + 31) / 32 * 32;
  const int grid = (int)((p.ncells + range - 1) / range);
  auto kern = k_assemble_tc_shift<FORM, D, PREC>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, H_THREADS, smem, s>>>(p, range);
  return cudaGetLastError();
}

template <int FORM, int D>
cudaError_t launch_shift_prec(const TcParams& p, int num_sms, cudaStream_t s, int smem) {
  switch (p.precision) {
    case PREC_TF32: return launch_shift_typed<FORM, D, PREC_TF32>(p, num_sms, s, smem);
    case PREC_TF32X3: return launch_shift_typed<FORM, D, PREC_TF32X3>(p, num_sms, s, smem);
    case PREC_BF16: return launch_shift_typed<FORM, D, PREC_BF16>(p, num_sms, s, smem);
    case PREC_BF16X3: return launch_shift_typed<FORM, D, PREC_BF16X3>(p, num_sms, s, smem);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

// Where this kernel runs: rows off the 32-byte sectors, matrices of more than one slice of 128 entries, and enough
// cells. us, this kernel / k_assemble_tc (tetrahedra P4, then triangles P4; mm MMAs an accumulator):
//             cells:  3001       20,011     65,536     200,001    524,288
//   tets mm = 1       26 / 20    28 / 36    60 / 111   186 / 354  456 / 982
//   tets mm = 3       32 / 20    33 / 35    61 / 118   164 / 361  381 / 977
//   tets mm = 6       40 / 21    42 / 37    78 / 116   215 / 362  493 / 985
//   tris mm = 1 or 2  9.0 / 7.5  9.5 / 10.8 15 / 17    35 / 43    83 / 120
//   tris mm = 3       10 / 7.6   11 / 11    17 / 17    40 / 43    86 / 125
//   tris mm = 6       12 / 7.8   13 / 11    21 / 18    50 / 40    109 / 93
// Few cells do not fill tiles of 256 in eight classes, and with few slices the MMAs take longer than the stores.
namespace {
struct ShiftShape {
  int mtiles, mm;  // slices of 128 entries, MMAs an accumulator
  bool fits;
};
ShiftShape shift_shape(int form, int degree, int cell, int precision) {
  const bool tf32 = precision == PREC_TF32 || precision == PREC_TF32X3;
  const int kstep = tf32 ? 8 : 16, K = form_K(form, degree, cell), ksteps = (K + kstep - 1) / kstep;
  const int ns = nnodes(cell, degree), N = ns * ns, mtiles = (N + BM - 1) / BM;
  const int passes = precision == PREC_TF32 ? 1 : precision == PREC_BF16 ? 2 : precision == PREC_TF32X3 ? 3 : 6;
  return {mtiles, ksteps * passes, mtiles > 1 && N + 7 <= mtiles * BM && shift_smem(mtiles, ksteps * 32, precision) <= 227 * 1024};
}
}  // namespace

// whether some count of cells and stride takes this kernel
int tc_shift_possible(int form, int degree, int cell, int precision) {
  if (!(form == FORM_MASS || form == FORM_HELMHOLTZ || form == FORM_ADVDIFF) || cell == CELL_PRISM || precision == PREC_FP64) return 0;
  const ShiftShape s = shift_shape(form, degree, cell, precision);
  return s.fits && !(s.mm > 3 && s.mtiles <= 4);
}

int tc_shift_use(int form, int degree, int cell, int precision, int64_t ostride, unsigned tune, int64_t ncells) {
  if (!tc_shift_possible(form, degree, cell, precision) || ostride % 8 == 0) return 0;
  if ((tune & TUNE_KNOBS) && !(tune & TUNE_HINT)) return 0;  // a knob of the other kernel's asks for that kernel
  const ShiftShape s = shift_shape(form, degree, cell, precision);
  return ncells >= (s.mtiles > 4 ? (s.mm > 3 ? 32768 : 16384) : s.mm == 3 ? 131072 : 16384);
}

void build_shift_image(int form, int degree, int cell, int prec, std::vector<uint8_t>& img) {
  std::vector<double> T;
  tc_reference_tensor(form, degree, cell, T);
  const bool tf32 = prec == PREC_TF32 || prec == PREC_TF32X3;
  const int elem = tf32 ? 4 : 2, kstep = tf32 ? 8 : 16, K = form_K(form, degree, cell);
  const int ns = nnodes(cell, degree), N = ns * ns, rows = (N + BM - 1) / BM * BM + 8;
  const size_t part = (size_t)rows * ((K + kstep - 1) / kstep * 32);
  img.assign(prec_tparts(prec) * part, 0);
  for (int o = 0; o < N; ++o)
    for (int k = 0; k < K; ++k)
      host_store_parts(img.data(), part, (uint32_t)((k * elem / 16 * rows + 8 + o) * 16 + k * elem % 16),
                       T[(size_t)k * N + o], tf32, prec_tparts(prec));
}

int launch_tc_shift(int form, int cell, const TcParams& p, int num_sms, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  TcParams q = p;
  q.image = p.shift_image;
  q.classes = (p.ostride & 1) ? 8 : (p.ostride & 2) ? 4 : 2;
  int smem = shift_smem(p.mtiles, p.kbytes, p.precision);
  if (smem < 120 * 1024) smem = 120 * 1024;  // one CTA (one owner of all TMEM columns) per SM
  const bool tri = cell == CELL_TRI;
  switch (form) {
    case FORM_MASS:
      return (int)(tri ? launch_shift_prec<FORM_MASS, 2>(q, num_sms, s, smem) : launch_shift_prec<FORM_MASS, 3>(q, num_sms, s, smem));
    case FORM_HELMHOLTZ:
      return (int)(tri ? launch_shift_prec<FORM_HELMHOLTZ, 2>(q, num_sms, s, smem)
                       : launch_shift_prec<FORM_HELMHOLTZ, 3>(q, num_sms, s, smem));
    case FORM_ADVDIFF:
      return (int)(tri ? launch_shift_prec<FORM_ADVDIFF, 2>(q, num_sms, s, smem)
                       : launch_shift_prec<FORM_ADVDIFF, 3>(q, num_sms, s, smem));
  }
  return (int)cudaErrorInvalidValue;
}

}  // namespace coffee
