// FP64 assembly on prisms: MASS, HELMHOLTZ and ADVDIFF, and vector Burgers (section 5.2 runs it on the third
// element shape as well): the Jacobian of
//   R[(c,i)] = int (u.grad u_c) phi_i + nu grad u_c . grad phi_i,
// or R itself.
//
// A prism's map x(xi) = sum_v N_v(xi) X_v (degree-1 prism functions) is not affine, so the Jacobian J, its
// determinant and K = J^-1 belong to the quadrature point and the element matrix stays a sum over points. But
// rule, basis and point set are products of triangle and interval, phi_(it,iz) = psi_it(s,t) zeta_iz(z), so the
// sum is taken in two steps. The forms are sums over points q = (qt, qz) of at most 18 factors,
//   M (scalar mass: w|det|; Burgers: w|det| d_cj u_ci, nine),   V_ab = w|det| (K K^T)_ab (times eps or nu),
//   beta_a = w|det| (K b)_a,   A_ij = sum_q M phi_i phi_j + V_ab d_a phi_i d_b phi_j + phi_i beta_a d_a phi_j:
// first, per triangle point and pair (iz <= jz), the factors are summed over qz against the products of
// zeta and zeta' (8 to 21 fields); then, per pair (it <= jt), over qt against the products of psi and its
// derivatives. One such quadruple gives the up to four entries that exchange it with jt and iz with jz, which
// differ only in signs once the products of psi and d psi are taken as half sums and differences (below).
//
// The FP64 pipe (2 FMAs per cycle and SM) bounds this as it did the sums over all points that stood here
// before (Burgers Jacobian P2: 435,000 FMAs a cell, 33.7 ms for 27,648 cells; Helmholtz P2 145,000). The two
// steps take 22 FMAs per quadruple and triangle point (Burgers; Helmholtz 8, advection-diffusion 13; with the
// exchanged entries summed one by one 27, 13, 18), 44,000 in all for P2 where the direct sum takes 21 per entry and
// point. u and its derivatives at the points are formed the same way.
// Measured, now / the exchanged entries one by one / the direct sums: Burgers Jacobian 27,648 P2 3.35 / 3.77 /
// 33.65 ms (44,000 + 9,000 FMAs), P1 0.40 ms for 20,000, 300 P4 1.16 ms; 27,648 P2 Helmholtz 1.29 / 1.74 /
// 7.62, advection-diffusion 1.97 / 2.40 / 9.81 ms. Now / the direct sums: residual P2 0.95 / 2.83, mass 0.31 / 1.24 ms;
// 60,000 P1 Helmholtz 0.58 / 1.74 ms; 300 cells P1 16-36 us as launched from Python against 33-81, P4 0.05-1.2 ms
// against 1.1-70.
// A block holds one cell (P1: seven, residual P2: two), its factors and fields in shared memory, and several
// blocks share an SM, so that one's table reads and barriers hide behind another's FMAs.
#include <cuda_runtime.h>
#include "coffee_internal.h"

namespace coffee {
namespace {

template <int FORM, int DEG>
struct Sf {
  static constexpr bool burgers = FORM == FORM_BURGERS || FORM == FORM_BURGERS_RES;
  static constexpr bool res = FORM == FORM_BURGERS_RES;
  static constexpr int P = burgers ? (3 * DEG + 3) / 2 : DEG + 2;  // points per direction
  static constexpr int QT = P * P, QZ = P, Q = QT * QZ;
  static constexpr int NT = (DEG + 1) * (DEG + 2) / 2, NZ = DEG + 1, n = NT * NZ, N = burgers ? 3 * n : n;
  static constexpr int NTP = NT * (NT + 1) / 2, NZP = NZ * (NZ + 1) / 2;
  static constexpr int NM = FORM == FORM_BURGERS ? 9 : FORM == FORM_ADVDIFF ? 0 : 1;  // M fields
  static constexpr bool V = FORM != FORM_MASS, BETA = FORM == FORM_ADVDIFF || FORM == FORM_BURGERS;
  static constexpr int NF = res ? 12 : NM + (V ? 6 : 0) + (BETA ? 3 : 0);              // factors of a point
  static constexpr int NB = NM == 9 ? 9 : 0;                                           // of them, a block's own (M)
  static constexpr int NFLD = res ? 9 : !V ? 1 : BETA ? NB + 11 : 8;                   // fields of (qt, z pair)
  static constexpr int items = res ? 3 * n : NTP * NZP;                                // of one cell, last step
  static constexpr int CELLS = DEG == 1 ? 7 : res && DEG == 2 ? 2 : 1;
  static constexpr int THREADS = DEG == 3 && !res ? 192 : DEG == 4 && !res ? 320 : 128;
  // doubles of shared memory per cell: factors, fields, vertices, node values, u along z
  static constexpr int S1 = QT * (res ? NZ : NZP) * NFLD;
  static constexpr int XU = 18 + (burgers ? 3 * n : 24), WZ = burgers ? 3 * NT * QZ * 2 : 0;
  static constexpr int cell_doubles = Q * NF + S1 + XU + WZ;
  static constexpr int ZTAB = QZ * NZP * 4 + QZ * NZ * 2;  // z products and zeta, zeta' (shared by the block)
  static constexpr size_t smem = sizeof(double) * ((size_t)CELLS * cell_doubles + ZTAB) + 16 * sizeof(int);
  // offsets in the host's table (prism_sum_table)
  static constexpr int T_PSI = 0, T_TP = T_PSI + QT * NT * 3, T_ZP = T_TP + QT * 12 * NTP, T_PT = T_ZP + ZTAB;
};

// Geometry at a point: adjugate (K = adj / det) and determinant
__device__ __forceinline__ double prism_geometry(const double* X, double s, double t, double z, double (&adj)[3][3]) {
  const double lam[3] = {1.0 - s - t, s, t};
  double J[3][3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    double mid[3], jz = 0.0;
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      const double lo = X[v * 3 + r], hi = X[(v + 3) * 3 + r];
      mid[v] = (1.0 - z) * lo + z * hi;
      jz += lam[v] * (hi - lo);
    }
    J[r][0] = mid[1] - mid[0];
    J[r][1] = mid[2] - mid[0];
    J[r][2] = jz;
  }
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const int r1 = (m + 1) % 3, r2 = (m + 2) % 3, a1 = (a + 1) % 3, a2 = (a + 2) % 3;
      adj[a][m] = J[r1][a1] * J[r2][a2] - J[r1][a2] * J[r2][a1];
    }
  return J[0][0] * adj[0][0] + J[0][1] * adj[1][0] + J[0][2] * adj[2][0];
}

template <int FORM, int DEG, bool CSR>
__global__ void __launch_bounds__(Sf<FORM, DEG>::THREADS) k_prism_sf(const PrismParams p) {
  using S = Sf<FORM, DEG>;
  constexpr int QT = S::QT, QZ = S::QZ, Q = S::Q, NT = S::NT, NZ = S::NZ, n = S::n, N = S::N, NF = S::NF, NFLD = S::NFLD,
                NTP = S::NTP, NZP = S::NZP, NM = S::NM, NB = S::NB, CELLS = S::CELLS, THREADS = S::THREADS;
  extern __shared__ double sm[];
  double* sF = sm;                                  // [CELLS][Q][NF]
  double* sS = sF + CELLS * Q * NF;                 // [CELLS][QT][NZP or NZ][NFLD]
  double* sX = sS + CELLS * S::S1;                  // [CELLS][18 vertices, then u [n][3] or (eps, b) [6][4]]
  double* sW = sX + CELLS * S::XU;                  // [CELLS][3][NT][QZ][2]: u along z, its derivative
  double* sZ = sW + CELLS * S::WZ;                  // z products [QZ][NZP][4], zeta and zeta' [QZ][NZ][2]
  int* sbad = reinterpret_cast<int*>(sZ + S::ZTAB);  // [CELLS]
  const int tid = threadIdx.x;
  const double* __restrict__ psi = p.T + S::T_PSI;  // [QT][NT][3]: psi, d_s, d_t
  const double* __restrict__ tp = p.T + S::T_TP;    // [QT][12][NTP]
  const double* __restrict__ pt = p.T + S::T_PT;    // triangle points [QT][3] (s, t, weight), z [QZ][2] (z, weight)
  for (int i = tid; i < S::ZTAB; i += THREADS) sZ[i] = __ldg(p.T + S::T_ZP + i);
  const double* zl = sZ + QZ * NZP * 4;

  for (int64_t e0 = (int64_t)blockIdx.x * CELLS; e0 < p.ncells; e0 += (int64_t)gridDim.x * CELLS) {
    const int nc = p.ncells - e0 < CELLS ? (int)(p.ncells - e0) : CELLS;
    __syncthreads();  // the cells before have been written
    if (tid < CELLS) sbad[tid] = 0;
    __syncthreads();
    // ---- vertices and coefficients ----
    for (int i = tid; i < nc * 18; i += THREADS) {
      const int c = i / 18, k = i % 18, vid = __ldg(p.c2v + (e0 + c) * 6 + k / 3);
      const bool bad = p.validate && (vid < 0 || vid >= p.nverts);
      if (bad) sbad[c] = 1;
      sX[c * S::XU + k] = bad ? 0.0 : __ldg(p.coords + (int64_t)vid * 3 + k % 3);
    }
    if constexpr (S::burgers || FORM == FORM_ADVDIFF) {
      constexpr int rows = S::burgers ? n : 6, w = S::burgers ? 3 : 4;
      for (int i = tid; i < nc * rows; i += THREADS) {
        const int c = i / rows, r = i % rows, id = __ldg(p.c2d + (e0 + c) * rows + r);
        const bool bad = p.validate && (id < 0 || id >= p.ncoefnodes);
        if (bad) sbad[c] = 1;
#pragma unroll
        for (int k = 0; k < w; ++k) sX[c * S::XU + 18 + r * w + k] = bad ? 0.0 : __ldg(p.coef + (int64_t)id * w + k);
      }
    }
    __syncthreads();
    if (tid < nc && sbad[tid]) atomicOr(p.err, ERR_INDEX);
    // ---- u and its z derivative on the triangle's nodes, at the z points ----
    if constexpr (S::burgers) {
      for (int i = tid; i < nc * 3 * NT * QZ; i += THREADS) {
        const int qz = i % QZ, it = i / QZ % NT, ch = i / (QZ * NT) % 3, c = i / (QZ * NT * 3);
        const double* U = sX + c * S::XU + 18;
        double v = 0.0, d = 0.0;
#pragma unroll
        for (int iz = 0; iz < NZ; ++iz) {
          const double u = U[(iz * NT + it) * 3 + ch];
          v = fma(u, zl[(qz * NZ + iz) * 2], v);
          d = fma(u, zl[(qz * NZ + iz) * 2 + 1], d);
        }
        double* w = sW + c * S::WZ + ((ch * NT + it) * QZ + qz) * 2;
        w[0] = v;
        w[1] = d;
      }
      __syncthreads();
    }
    // ---- the factors at every point ----
    for (int i = tid; i < nc * Q; i += THREADS) {
      const int c = i / Q, q = i % Q, qt = q / QZ, qz = q % QZ;
      const double s = __ldg(pt + qt * 3), t = __ldg(pt + qt * 3 + 1), z = __ldg(pt + QT * 3 + qz * 2);
      const double wq = __ldg(pt + qt * 3 + 2) * __ldg(pt + QT * 3 + qz * 2 + 1);
      double adj[3][3];
      const double det = prism_geometry(sX + c * S::XU, s, t, z, adj);
      const double ad = fabs(det), sg = det < 0.0 ? -wq : wq;
      double* f = sF + (size_t)(c * Q + q) * NF;
      if constexpr (FORM == FORM_MASS || FORM == FORM_HELMHOLTZ) f[0] = wq * ad;
      double vs = wq / ad;  // w|det| K K^T = w adj adj^T / |det|
      double b[3] = {0.0, 0.0, 0.0};
      if constexpr (FORM == FORM_ADVDIFF) {
        const double* cf = sX + c * S::XU + 18;
        const double lam[3] = {1.0 - s - t, s, t};
        double eps = 0.0;
#pragma unroll
        for (int v = 0; v < 6; ++v) {
          const double Nv = v < 3 ? lam[v % 3] * (1.0 - z) : lam[v % 3] * z;
          eps += Nv * cf[v * 4];
#pragma unroll
          for (int r = 0; r < 3; ++r) b[r] += Nv * cf[v * 4 + 1 + r];
        }
        vs *= eps;
      }
      if constexpr (S::burgers) {
        // u and its reference gradient, then w|det| times the physical gradient: w sign(det) adj^T grad
        double uq[3] = {0.0, 0.0, 0.0}, gr[3][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
        for (int it = 0; it < NT; ++it) {
          const double* ps = psi + (qt * NT + it) * 3;
          const double p0 = __ldg(ps), p1 = __ldg(ps + 1), p2 = __ldg(ps + 2);
#pragma unroll
          for (int ch = 0; ch < 3; ++ch) {
            const double* w = sW + c * S::WZ + ((ch * NT + it) * QZ + qz) * 2;
            uq[ch] = fma(p0, w[0], uq[ch]);
            gr[ch][0] = fma(p1, w[0], gr[ch][0]);
            gr[ch][1] = fma(p2, w[0], gr[ch][1]);
            gr[ch][2] = fma(p0, w[1], gr[ch][2]);
          }
        }
        vs *= p.nu;
        if constexpr (!S::res) {
#pragma unroll
          for (int ci = 0; ci < 3; ++ci)
#pragma unroll
            for (int cj = 0; cj < 3; ++cj)
              f[ci * 3 + cj] = sg * (adj[0][cj] * gr[ci][0] + adj[1][cj] * gr[ci][1] + adj[2][cj] * gr[ci][2]);
#pragma unroll
          for (int r = 0; r < 3; ++r) b[r] = uq[r];
        } else {
          double y[3];  // sign(det) w adj u: (u.grad u_c) = y . reference gradient
#pragma unroll
          for (int a = 0; a < 3; ++a) y[a] = sg * (adj[a][0] * uq[0] + adj[a][1] * uq[1] + adj[a][2] * uq[2]);
          double H[6];
          int k = 0;
#pragma unroll
          for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int e = a; e < 3; ++e)
              H[k++] = vs * (adj[a][0] * adj[e][0] + adj[a][1] * adj[e][1] + adj[a][2] * adj[e][2]);
#pragma unroll
          for (int ch = 0; ch < 3; ++ch) {
            f[ch] = y[0] * gr[ch][0] + y[1] * gr[ch][1] + y[2] * gr[ch][2];
            f[3 + ch * 3] = H[0] * gr[ch][0] + H[1] * gr[ch][1] + H[2] * gr[ch][2];
            f[3 + ch * 3 + 1] = H[1] * gr[ch][0] + H[3] * gr[ch][1] + H[4] * gr[ch][2];
            f[3 + ch * 3 + 2] = H[2] * gr[ch][0] + H[4] * gr[ch][1] + H[5] * gr[ch][2];
          }
        }
      }
      if constexpr (S::V && !S::res) {
        int k = NM;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int e = a; e < 3; ++e)
            f[k++] = vs * (adj[a][0] * adj[e][0] + adj[a][1] * adj[e][1] + adj[a][2] * adj[e][2]);
      }
      if constexpr (S::BETA) {
#pragma unroll
        for (int a = 0; a < 3; ++a) f[NM + 6 + a] = sg * (adj[a][0] * b[0] + adj[a][1] * b[1] + adj[a][2] * b[2]);
      }
    }
    __syncthreads();
    if constexpr (!S::res) {
      // ---- sums over z of M zeta_i zeta_j, V_ss, V_st, V_tt (zeta_i zeta_j), V_zz (zeta'_i zeta'_j), V_sz and V_tz
      // with zeta_i zeta'_j (1) and with zeta_j zeta'_i (2), beta_s, beta_t (zeta_i zeta_j), beta_z (1, 2); of these
      // the fields, in the order of the tables they meet below ----
      for (int i = tid; i < nc * QT * NZP; i += THREADS) {
        const int zp = i % NZP, qt = i / NZP % QT, c = i / (NZP * QT);
        double m[NM > 0 ? NM : 1], ss = 0.0, st = 0.0, tt = 0.0, zz = 0.0, sz1 = 0.0, sz2 = 0.0, tz1 = 0.0, tz2 = 0.0,
               bs = 0.0, bt = 0.0, bz1 = 0.0, bz2 = 0.0;
#pragma unroll
        for (int k = 0; k < (NM > 0 ? NM : 1); ++k) m[k] = 0.0;
        const double* f = sF + (size_t)(c * Q + qt * QZ) * NF;
#pragma unroll 2
        for (int qz = 0; qz < QZ; ++qz, f += NF) {
          const double* w = sZ + (qz * NZP + zp) * 4;
          const double w0 = w[0], w1 = w[1], w2 = w[2], w3 = w[3];
#pragma unroll
          for (int k = 0; k < NM; ++k) m[k] = fma(f[k], w0, m[k]);
          if constexpr (S::V) {  // pairs ss, st, sz, tt, tz, zz
            ss = fma(f[NM], w0, ss);
            st = fma(f[NM + 1], w0, st);
            tt = fma(f[NM + 3], w0, tt);
            zz = fma(f[NM + 5], w3, zz);
            sz1 = fma(f[NM + 2], w1, sz1);
            sz2 = fma(f[NM + 2], w2, sz2);
            tz1 = fma(f[NM + 4], w1, tz1);
            tz2 = fma(f[NM + 4], w2, tz2);
          }
          if constexpr (S::BETA) {
            bs = fma(f[NM + 6], w0, bs);
            bt = fma(f[NM + 7], w0, bt);
            bz1 = fma(f[NM + 8], w1, bz1);
            bz2 = fma(f[NM + 8], w2, bz2);
          }
        }
        double* o = sS + c * S::S1 + (qt * NZP + zp) * NFLD;
        if constexpr (!S::V) {
          o[0] = m[0];
        } else {
#pragma unroll
          for (int k = 0; k < NB; ++k) o[k] = m[k];
          o += NB;
          o[0] = ss, o[1] = st, o[2] = tt;
          o[3] = sz1 + sz2, o[4] = tz1 + tz2;
          o[5] = sz1 - sz2, o[6] = tz1 - tz2;
          if constexpr (S::BETA) {
            o[7] = bs, o[8] = bt;
            o[9] = zz + bz1, o[10] = zz + bz2;
          } else {
            o[7] = zz + m[0];
          }
        }
      }
      __syncthreads();
      // ---- sums over the triangle's points, one quadruple (it <= jt, iz <= jz) per thread. Exchanging it with jt
      // leaves P+, R+ = (d psi_it psi_jt + psi_it d psi_jt) / 2 as they are and turns the sign of P-, R-; exchanging
      // iz with jz turns that of V_sz, V_tz (1) - (2). So the four entries are
      //   C +- G + v1 + y    and    C -+ G + v2 + y,   G = sum (sz1 - sz2) P- + (tz1 - tz2) R-,
      // C the sum of the ss, st, tt terms and of (sz1 + sz2) P+ + (tz1 + tz2) R+, common to all. What a half sum adds
      // and the difference takes away again, sz1 psi_it d psi_jt and so on, is of the size of the terms of V_sz that the
      // entry has (the ratio is one of basis functions). The flow's terms y are no such pair: an entry has either
      // beta_s d psi_it psi_jt or beta_s psi_it d psi_jt (y2, y1), and one of these may be zero (flow along an axis), so
      // they are summed each (with half sums of them too, 3.18 ms for 3.35 of the Burgers Jacobian P2, entries of the diffusion alone were
      // off by roundings of the flow's). ----
      for (int i = tid; i < nc * S::items; i += THREADS) {
        const int c = i / S::items, k = i % S::items, zp = k / NTP, tq = k % NTP;
        double M[NB > 0 ? NB : 1], C = 0.0, G = 0.0, v1 = 0.0, v2 = 0.0, y1 = 0.0, y2 = 0.0;
#pragma unroll
        for (int x = 0; x < (NB > 0 ? NB : 1); ++x) M[x] = 0.0;
        const double* f = sS + c * S::S1 + zp * NFLD;
        const double* tt = tp + tq;
#pragma unroll 2
        for (int qt = 0; qt < QT; ++qt, f += NZP * NFLD, tt += 12 * NTP) {
          const double T = __ldg(tt);
#pragma unroll
          for (int x = 0; x < NB; ++x) M[x] = fma(f[x], T, M[x]);
          if constexpr (S::V) {
            const double* h = f + NB;
            const double Pp = __ldg(tt + 4 * NTP), Pm = __ldg(tt + 5 * NTP), Rp = __ldg(tt + 6 * NTP), Rm = __ldg(tt + 7 * NTP);
            C = fma(h[0], __ldg(tt + NTP), fma(h[1], __ldg(tt + 2 * NTP), fma(h[2], __ldg(tt + 3 * NTP), C)));
            C = fma(h[3], Pp, fma(h[4], Rp, C));
            G = fma(h[5], Pm, fma(h[6], Rm, G));
            if constexpr (S::BETA) {
              y1 = fma(h[7], __ldg(tt + 9 * NTP), fma(h[8], __ldg(tt + 11 * NTP), y1));
              y2 = fma(h[7], __ldg(tt + 8 * NTP), fma(h[8], __ldg(tt + 10 * NTP), y2));
              v1 = fma(h[9], T, v1);
              v2 = fma(h[10], T, v2);
            } else {
              C = fma(h[7], T, C);
            }
          } else {
            C = fma(f[0], T, C);
          }
        }
        if (sbad[c]) continue;
        int jt = 0, jz = 0;  // tq = jt (jt + 1) / 2 + it, zp = jz (jz + 1) / 2 + iz
        while ((jt + 1) * (jt + 2) / 2 <= tq) ++jt;
        while ((jz + 1) * (jz + 2) / 2 <= zp) ++jz;
        const int it = tq - jt * (jt + 1) / 2, iz = zp - jz * (jz + 1) / 2;
        const int64_t e = e0 + c;
        auto put = [&](int row, int col, double d) {  // d: the terms of the diagonal blocks
#pragma unroll
          for (int ci = 0; ci < (S::burgers ? 3 : 1); ++ci)
#pragma unroll
            for (int cj = 0; cj < (S::burgers ? 3 : 1); ++cj) {
              const int at = (ci * n + row) * N + cj * n + col;
              double v = ci == cj ? d : 0.0;
              if constexpr (NB > 0) v += M[ci * 3 + cj];
              if constexpr (CSR) {
                const uint32_t pos = __ldg(p.map + csr_map_index(e, at, (N * N + 3) & ~3));
                if (pos < (uint64_t)p.nnz) atomicAdd(static_cast<double*>(p.out) + pos, v);
                else atomicOr(p.err, ERR_INDEX);
              } else {
                static_cast<double*>(p.out)[e * (int64_t)(N * N) + at] = v;
              }
            }
        };
        put(iz * NT + it, jz * NT + jt, (C + G) + (v1 + y1));
        if (it != jt) put(iz * NT + jt, jz * NT + it, (C - G) + (v1 + y2));
        if (iz != jz) put(jz * NT + it, iz * NT + jt, (C - G) + (v2 + y1));
        if (it != jt && iz != jz) put(jz * NT + jt, iz * NT + it, (C + G) + (v2 + y2));
      }
    } else {
      // ---- residual: sums over z of a_c zeta + gamma_cz zeta', gamma_cs zeta, gamma_ct zeta, then over qt ----
      for (int i = tid; i < nc * QT * NZ; i += THREADS) {
        const int iz = i % NZ, qt = i / NZ % QT, c = i / (NZ * QT);
        double a[9] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        const double* f = sF + (size_t)(c * Q + qt * QZ) * NF;
#pragma unroll 2
        for (int qz = 0; qz < QZ; ++qz, f += NF) {
          const double w0 = zl[(qz * NZ + iz) * 2], w1 = zl[(qz * NZ + iz) * 2 + 1];
#pragma unroll
          for (int ch = 0; ch < 3; ++ch) {
            a[ch * 3] = fma(f[ch], w0, fma(f[3 + ch * 3 + 2], w1, a[ch * 3]));
            a[ch * 3 + 1] = fma(f[3 + ch * 3], w0, a[ch * 3 + 1]);
            a[ch * 3 + 2] = fma(f[3 + ch * 3 + 1], w0, a[ch * 3 + 2]);
          }
        }
        double* o = sS + c * S::S1 + (qt * NZ + iz) * 9;
#pragma unroll
        for (int k = 0; k < 9; ++k) o[k] = a[k];
      }
      __syncthreads();
      for (int i = tid; i < nc * S::items; i += THREADS) {
        const int c = i / S::items, k = i % S::items, ch = k / n, node = k % n, iz = node / NT, it = node % NT;
        const double* f = sS + c * S::S1 + iz * 9 + ch * 3;
        double acc = 0.0;
#pragma unroll 2
        for (int qt = 0; qt < QT; ++qt, f += NZ * 9) {
          const double* ps = psi + (qt * NT + it) * 3;
          acc = fma(f[0], __ldg(ps), fma(f[1], __ldg(ps + 1), fma(f[2], __ldg(ps + 2), acc)));
        }
        if (!sbad[c]) static_cast<double*>(p.out)[(e0 + c) * (int64_t)N + k] = acc;
      }
    }
  }
}

template <int FORM, int DEG>
cudaError_t launch_sf(const PrismParams& p, int num_sms, cudaStream_t s) {
  using S = Sf<FORM, DEG>;
  if (p.Q != S::Q) return cudaErrorInvalidValue;
  const int64_t blocks = (p.ncells + S::CELLS - 1) / S::CELLS;
  const unsigned grid = (unsigned)(blocks < (int64_t)num_sms * 16 ? blocks : (int64_t)num_sms * 16);
  auto go = [&](auto kern) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, S::THREADS, S::smem, s>>>(p);
    return cudaGetLastError();
  };
  if constexpr (!S::res)
    if (p.map) return go(k_prism_sf<FORM, DEG, true>);
  return go(k_prism_sf<FORM, DEG, false>);
}

template <int FORM>
cudaError_t launch_sf_deg(int degree, const PrismParams& p, int num_sms, cudaStream_t s) {
  switch (degree) {
    case 1: return launch_sf<FORM, 1>(p, num_sms, s);
    case 2: return launch_sf<FORM, 2>(p, num_sms, s);
    case 3: return launch_sf<FORM, 3>(p, num_sms, s);
    case 4: return launch_sf<FORM, 4>(p, num_sms, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

int launch_prism(int form, int degree, const PrismParams& p, int num_sms, void* stream) {
  if (p.ncells == 0) return (int)cudaSuccess;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  switch (form) {
    case FORM_MASS: return (int)launch_sf_deg<FORM_MASS>(degree, p, num_sms, s);
    case FORM_HELMHOLTZ: return (int)launch_sf_deg<FORM_HELMHOLTZ>(degree, p, num_sms, s);
    case FORM_ADVDIFF: return (int)launch_sf_deg<FORM_ADVDIFF>(degree, p, num_sms, s);
    case FORM_BURGERS: return (int)launch_sf_deg<FORM_BURGERS>(degree, p, num_sms, s);
    case FORM_BURGERS_RES: return (int)launch_sf_deg<FORM_BURGERS_RES>(degree, p, num_sms, s);
  }
  return (int)cudaErrorInvalidValue;
}

}  // namespace coffee
