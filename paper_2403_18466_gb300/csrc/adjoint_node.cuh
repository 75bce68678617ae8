// adjoint_node.cuh -- per-node pieces of the reverse mode shared by the FP32 and
// the tensor-core adjoint: the conservation projector and the vector-Jacobian
// products of the equilibrium.
#pragma once
#include "lattice.cuh"

namespace lbm {

__device__ __forceinline__ void project9(float o[Q]) {
  float s = 0.f, sx = 0.f, sy = 0.f;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    s += o[i];
    sx += (float)cx(i) * o[i];
    sy += (float)cy(i) * o[i];
  }
  const float k1 = -s * (1.0f / 9.0f), k2 = -sx * (1.0f / 6.0f), k3 = -sy * (1.0f / 6.0f);
#pragma unroll
  for (int i = 0; i < Q; ++i) o[i] += k1 + (float)cx(i) * k2 + (float)cy(i) * k3;
}

// Sums of a per-direction vector g against the partial derivatives of
// feq_i(rho, u) = w_i rho (1 + 3 c.u + 4.5 (c.u)^2 - 1.5 |u|^2).  feq_i is
// quadratic in c_i, so every such sum is a combination of the six weighted
// moments sum_i w_i g_i c_i^a c_i^b (monomials 1, c_x, c_y, c_x^2, c_x c_y,
// c_y^2): about 40 operations for the moments and 25 per velocity, instead of
// the 9 x 20 of a sum over directions.
struct GMom {
  float g0, gx, gy, gxx, gxy, gyy;
};
// Adds w_i g times the monomials of direction i (compile-time i).
__device__ __forceinline__ void gmom_add(GMom &s, int i, float g) {
  const float v = wf(i) * g;
  s.g0 += v;
  if (cx(i) != 0) {
    s.gx += cx(i) > 0 ? v : -v;
    s.gxx += v;
  }
  if (cy(i) != 0) {
    s.gy += cy(i) > 0 ? v : -v;
    s.gyy += v;
  }
  if (cx(i) * cy(i) != 0) s.gxy += cx(i) * cy(i) > 0 ? v : -v;
}
__device__ __forceinline__ GMom weighted_moments(const float g[Q]) {
  GMom s = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int i = 0; i < Q; ++i) gmom_add(s, i, g[i]);
  return s;
}
// sum_i g_i dfeq_i/drho, dfeq_i/du_x, dfeq_i/du_y at (rho, ux, uy)
__device__ __forceinline__ void feq_vjp(const GMom &s, float rho, float ux, float uy, float &sr,
                                        float &sx, float &sy) {
  const float usq = ux * ux + uy * uy;
  sr = s.g0 * (1.0f - 1.5f * usq) + 3.0f * (ux * s.gx + uy * s.gy) +
       4.5f * (ux * ux * s.gxx + 2.0f * ux * uy * s.gxy + uy * uy * s.gyy);
  sx = rho * (3.0f * s.gx + 9.0f * (ux * s.gxx + uy * s.gxy) - 3.0f * ux * s.g0);
  sy = rho * (3.0f * s.gy + 9.0f * (ux * s.gxy + uy * s.gyy) - 3.0f * uy * s.g0);
}

}  // namespace lbm
