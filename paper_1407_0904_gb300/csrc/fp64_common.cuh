// Per-cell geometry and factors of MASS, HELMHOLTZ and ADVDIFF in FP64, shared by the plain kernel
// (k_fp64.cu) and the tensor-core one (k_fp64_tc.cu).
#pragma once
#include <cuda_runtime.h>
#include <cstdint>
#include "coffee_internal.h"

namespace coffee {
namespace {

template <int D>
struct Geo {
  double adj[D][D];  // adjugate: K = adj / det
  double det;
};

template <int D>
__device__ __forceinline__ void geometry64(const double (&X)[D + 1][D], Geo<D>& g) {
  double J[D][D];
#pragma unroll
  for (int r = 0; r < D; ++r)
#pragma unroll
    for (int c = 0; c < D; ++c) J[r][c] = X[c + 1][r] - X[0][r];
  if constexpr (D == 2) {
    g.det = J[0][0] * J[1][1] - J[0][1] * J[1][0];
    g.adj[0][0] = J[1][1];
    g.adj[0][1] = -J[0][1];
    g.adj[1][0] = -J[1][0];
    g.adj[1][1] = J[0][0];
  } else {
    // cofactors C[r][c]; adj[a][r] = C[r][a]
    double C00 = J[1][1] * J[2][2] - J[1][2] * J[2][1];
    double C01 = J[1][2] * J[2][0] - J[1][0] * J[2][2];
    double C02 = J[1][0] * J[2][1] - J[1][1] * J[2][0];
    double C10 = J[0][2] * J[2][1] - J[0][1] * J[2][2];
    double C11 = J[0][0] * J[2][2] - J[0][2] * J[2][0];
    double C12 = J[0][1] * J[2][0] - J[0][0] * J[2][1];
    double C20 = J[0][1] * J[1][2] - J[0][2] * J[1][1];
    double C21 = J[0][2] * J[1][0] - J[0][0] * J[1][2];
    double C22 = J[0][0] * J[1][1] - J[0][1] * J[1][0];
    g.det = J[0][0] * C00 + J[0][1] * C01 + J[0][2] * C02;
    g.adj[0][0] = C00; g.adj[0][1] = C10; g.adj[0][2] = C20;
    g.adj[1][0] = C01; g.adj[1][1] = C11; g.adj[1][2] = C21;
    g.adj[2][0] = C02; g.adj[2][1] = C12; g.adj[2][2] = C22;
  }
}

template <int FORM, int D>
struct FormK {
  static constexpr int P = D * (D + 1) / 2;
  static constexpr int value = FORM == FORM_MASS ? 1
                               : FORM == FORM_HELMHOLTZ ? 1 + P
                               : FORM == FORM_ADVDIFF ? (D + 1) * P + (D + 1) * D
                                                      : 1;
};

// The kind of term of factor k, 0 or 1 (factors of one kind have one order of magnitude): mass and
// stiffness for HELMHOLTZ, stiffness and advection for ADVDIFF.
template <int FORM, int D>
__host__ __device__ constexpr int term_of(int k) {
  return FORM == FORM_HELMHOLTZ ? (k > 0) : FORM == FORM_ADVDIFF ? (k >= (D + 1) * FormK<FORM, D>::P) : 0;
}

// The factors of a cell: G[0..K) themselves, for ADVDIFF what they are products of: H (pairs a <= b), eps of the vertices, and
// the advection terms (22 numbers for 36 factors on tetrahedra, which a thread can keep in registers).
template <int FORM, int D>
struct Factors {
  static constexpr int NV = D + 1, P = D * (D + 1) / 2, K = FormK<FORM, D>::value;
  static constexpr int COUNT = FORM == FORM_ADVDIFF ? P + NV + NV * D : K;
  double f[COUNT];
  __device__ __forceinline__ double at(int k) const {
    if constexpr (FORM == FORM_ADVDIFF) return k < NV * P ? f[P + k / P] * f[k % P] : f[P + NV + k - NV * P];
    else return f[k];
  }
};

// The factors of cell e, false where an index is out of range (with p.validate). FAST: the
// division by |det| as one reciprocal and a corrected product each (q + (s - q |det|) / |det|, which is
// rounded as the division is but for rare last bits), instead of a division of about 20 instructions
// per pair.
template <int FORM, int D, bool FAST>
__device__ __forceinline__ bool factors64(const Fp64Params& p, int64_t e, Factors<FORM, D>& G) {
  constexpr int NV = D + 1, P = D * (D + 1) / 2;
  int vid[NV], cid[NV];
  bool bad = false;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    vid[v] = __ldg(p.c2v + e * NV + v);
    if (p.validate && (vid[v] < 0 || vid[v] >= p.nverts)) bad = true;
  }
  if constexpr (FORM == FORM_ADVDIFF) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      cid[v] = __ldg(p.c2d + e * NV + v);
      if (p.validate && (cid[v] < 0 || cid[v] >= p.ncoefnodes)) bad = true;
    }
  }
  if (bad) return false;
  double cf[FORM == FORM_ADVDIFF ? NV : 1][D + 1];  // (eps, b) of the vertices' nodes
  if constexpr (FORM == FORM_ADVDIFF) {
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int r = 0; r <= D; ++r) cf[v][r] = __ldg(p.coef + (int64_t)cid[v] * (D + 1) + r);
  }
  double X[NV][D];
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int r = 0; r < D; ++r) X[v][r] = __ldg(p.coords + (int64_t)vid[v] * D + r);
  Geo<D> g;
  geometry64<D>(X, g);
  const double Dm = fabs(g.det);
  if constexpr (FORM == FORM_MASS) {
    G.f[0] = Dm;
  } else {
    double H[P];  // |det| (K K^T)_{ab} = (adj adj^T)_{ab} / |det|, pairs a <= b
    const double inv = FAST ? 1.0 / Dm : 0.0;
    int q = 0;
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
      for (int b = a; b < D; ++b) {
        double s = 0.0;
#pragma unroll
        for (int r = 0; r < D; ++r) s += g.adj[a][r] * g.adj[b][r];
        if constexpr (FAST) {
          const double h = s * inv;
          H[q++] = fma(fma(-h, Dm, s), inv, h);
        } else {
          H[q++] = s / Dm;
        }
      }
    if constexpr (FORM == FORM_HELMHOLTZ) {
      G.f[0] = Dm;
#pragma unroll
      for (int k = 0; k < P; ++k) G.f[1 + k] = H[k];
    } else {
      const double sg = g.det < 0.0 ? -1.0 : 1.0;
#pragma unroll
      for (int k = 0; k < P; ++k) G.f[k] = H[k];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        G.f[P + v] = cf[v][0];
#pragma unroll
        for (int a = 0; a < D; ++a) {
          double s = 0.0;
#pragma unroll
          for (int r = 0; r < D; ++r) s += (sg * g.adj[a][r]) * cf[v][1 + r];
          G.f[P + NV + v * D + a] = s;
        }
      }
    }
  }
  return true;
}

}  // namespace
}  // namespace coffee
