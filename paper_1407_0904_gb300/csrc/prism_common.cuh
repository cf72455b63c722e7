// FP32 factors of prisms at a point, shared by the tensor-core kernels (k_prism_tc.cu, k_prism_sum_tc.cu).
#pragma once
#include <cuda_runtime.h>

namespace coffee {
namespace {

// Factors of one quadrature point pq = (s, t, z, w) of a prism, |det J| (1, (K K^T)_ab) or |det J| (eps (K K^T)_ab,
// (K b)_a): J from the per-cell bilinear coefficients (d/ds = A + z B, d/dt = C + z D, d/dz = E + s F + t G), and for
// advection-diffusion eps and b from the six vertex values CF. Every factor is linear in w.
template <int KQ>
__device__ __forceinline__ void prism_point_factors(const float4 pq, const float (&JA)[3], const float (&JB)[3],
                                                    const float (&JC)[3], const float (&JD)[3], const float (&JE)[3],
                                                    const float (&JF)[3], const float (&JG)[3],
                                                    const float (&CF)[6][4], float (&gf)[9]) {
  float J[3][3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    J[r][0] = fmaf(pq.z, JB[r], JA[r]);
    J[r][1] = fmaf(pq.z, JD[r], JC[r]);
    J[r][2] = fmaf(pq.x, JF[r], fmaf(pq.y, JG[r], JE[r]));
  }
  const float adj[3][3] = {{J[1][1] * J[2][2] - J[1][2] * J[2][1], J[0][2] * J[2][1] - J[0][1] * J[2][2],
                            J[0][1] * J[1][2] - J[0][2] * J[1][1]},
                           {J[1][2] * J[2][0] - J[1][0] * J[2][2], J[0][0] * J[2][2] - J[0][2] * J[2][0],
                            J[0][2] * J[1][0] - J[0][0] * J[1][2]},
                           {J[1][0] * J[2][1] - J[1][1] * J[2][0], J[0][1] * J[2][0] - J[0][0] * J[2][1],
                            J[0][0] * J[1][1] - J[0][1] * J[1][0]}};
  const float det = J[0][0] * adj[0][0] + J[0][1] * adj[1][0] + J[0][2] * adj[2][0];
  const float adet = fabsf(det);
  float wi = pq.w / adet;
  constexpr int P0 = KQ == 9 ? 0 : 1;  // first pair factor
  if constexpr (KQ == 9) {
    // eps and b at the point from the vertex values (degree-1 prism functions)
    const float lam[3] = {1.f - pq.x - pq.y, pq.x, pq.y};
    float eps = 0.f, bq[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      const float Nv = v < 3 ? lam[v] * (1.f - pq.z) : lam[v - 3] * pq.z;
      eps = fmaf(Nv, CF[v][0], eps);
#pragma unroll
      for (int r = 0; r < 3; ++r) bq[r] = fmaf(Nv, CF[v][1 + r], bq[r]);
    }
    const float sw = det < 0.f ? -pq.w : pq.w;
#pragma unroll
    for (int a = 0; a < 3; ++a) gf[6 + a] = sw * (adj[a][0] * bq[0] + adj[a][1] * bq[1] + adj[a][2] * bq[2]);
    wi *= eps;
  } else {
    gf[0] = pq.w * adet;
  }
  if constexpr (KQ > 1) {
#pragma unroll
    for (int a = 0, pp = P0; a < 3; ++a)
#pragma unroll
      for (int b = a; b < 3; ++b, ++pp) {
        float acc = 0.f;
#pragma unroll
        for (int r = 0; r < 3; ++r) acc = fmaf(adj[a][r], adj[b][r], acc);
        gf[pp] = wi * acc;
      }
  }
}

}  // namespace
}  // namespace coffee
