// d3q19_step.cu -- the paper's 3D setting on the CUDA cores: the fused D3Q19
// pull-stream + BGK / Smagorinsky-BGK step with the paper's three-component sine
// forcing (EDM, Eq. S5), and the data-movement kernels around it.
//
// Step kernels: one thread per node along x; each pulls f_i(x) = g_i(x - c_i)
// (periodic) from the previous buffer, collides and stores at x.  Algorithmic
// traffic 76 B read + 76 B written per node, which bounds them: measured (GB300,
// BGK / Smagorinsky) 45.6 / 45.4 G nodes/s at 256^3 and 43.4 / 43.2 at 128^3,
// against 43.6 / 40.1 and 41.2 / 38.0 with 64-bit wrapped addresses and the
// collision direction by direction (80 % of the issue slots).
#include <type_traits>

#include "approx.cuh"
#include "d3q19.cuh"
#include "kernels3d.h"
#include "umma.cuh"

namespace lbm {
namespace d3 {
namespace {

constexpr int NT = 128;

// f(0), ..., f(8) with compile-time arguments
template <class F>
__device__ __forceinline__ void each_pair(F &f) {
  f(std::integral_constant<int, 0>());
  f(std::integral_constant<int, 1>());
  f(std::integral_constant<int, 2>());
  f(std::integral_constant<int, 3>());
  f(std::integral_constant<int, 4>());
  f(std::integral_constant<int, 5>());
  f(std::integral_constant<int, 6>());
  f(std::integral_constant<int, 7>());
  f(std::integral_constant<int, 8>());
}
enum { KIND_BGK = 0, KIND_SMAG = 1 };

__device__ __forceinline__ int wrapi(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

struct Pos {
  int x, y, z, b;
};

__device__ __forceinline__ bool node_pos(const Grid3 &g, Pos &p) {
  p.x = blockIdx.x * NT + threadIdx.x;
  p.y = blockIdx.y;
  p.z = blockIdx.z % g.nz;
  p.b = blockIdx.z / g.nz;
  return p.x < g.nx;
}

__device__ __forceinline__ void pull(const float *__restrict__ in, const Grid3 &g, const Pos &p,
                                     float d[Q]) {
  const size_t vol = g.volume();
  const float *gb = in + (size_t)p.b * Q * vol;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int xs = wrapi(p.x - cx(i), g.nx), ys = wrapi(p.y - cy(i), g.ny),
              zs = wrapi(p.z - cz(i), g.nz);
    d[i] = __ldg(gb + (size_t)i * vol + ((size_t)zs * g.ny + ys) * g.nx + xs);
  }
}

__device__ __forceinline__ size_t at(const Grid3 &g, const Pos &p) {
  return ((size_t)p.z * g.ny + p.y) * g.nx + p.x;
}

__device__ __forceinline__ void node_force(const Collide3 &c, const Pos &p, float &Fx, float &Fy,
                                           float &Fz) {
  Fx = c.fx_y ? c.fx_y[p.y] : 0.f;
  Fy = c.fy_z ? c.fy_z[p.z] : 0.f;
  Fz = c.fz_x ? c.fz_x[p.x] : 0.f;
}

__device__ __forceinline__ void flag_bad(bool bad, int *flag) {
  const unsigned mask = __ballot_sync(__activemask(), bad);
  if (mask && (threadIdx.x & 31) == (unsigned)(__ffs(mask) - 1)) {
    if (*reinterpret_cast<volatile int *>(flag) == 0) atomicOr(flag, 1);
  }
}

// The nine directions with c > 0 of an opposite pair (their opposites are 7 - i
// for 4..6 and 25 - i for 13..18).
__host__ __device__ constexpr int pos_dir(int k) { return k < 3 ? 6 - k : 21 - k; }
__host__ __device__ constexpr int opposite(int i) { return i < 7 ? 7 - i : 25 - i; }
template <int K>
__device__ __forceinline__ float along(float ax, float ay, float az) {  // c . a
  constexpr int i = pos_dir(K);
  float r = 0.f;
  if (cx(i)) r = cx(i) > 0 ? ax : -ax;
  if (cy(i)) r = cx(i) ? (cy(i) > 0 ? r + ay : r - ay) : (cy(i) > 0 ? ay : -ay);
  if (cz(i)) r = cx(i) || cy(i) ? (cz(i) > 0 ? r + az : r - az) : (cz(i) > 0 ? az : -az);
  return r;
}

// Collide one node in place and add the force, on the even and odd parts
// s = f_i + f_opp, t = f_i - f_opp of the nine opposite pairs.  feq's even part is
// w E with E = drho - 1.5 j.u + 4.5 (c.j)(c.u), its odd part 3 w c.j, so a pair
// shares E, the stress of the Smagorinsky collision needs the even parts alone,
// and the EDM term (Eq. S5) has even part w (4.5 (c.F)(c.s_F) - 1.5 F.s_F),
// s_F = 2 u + F/rho, and odd part 3 w c.F: little more than half the operations of
// a sum direction by direction.  The weights multiply last: with 3 w as a rounded
// constant the momentum drifted by its error in every step (error against 64 bits
// after 20 steps at 128^3 4.7e-8 instead of 3.1e-8).  Returns true if the node is unstable.
template <int KIND>
__device__ __forceinline__ bool collide_pairs(float d[Q], const Collide3 &c, float Fx, float Fy,
                                              float Fz) {
  float s[9], t[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int i = pos_dir(k), o = opposite(i);
    s[k] = d[i] + d[o];
    t[k] = d[i] - d[o];
  }
  float drho = d[0], jx = 0.f, jy = 0.f, jz = 0.f;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int i = pos_dir(k);
    drho += s[k];
    if (cx(i)) jx += cx(i) > 0 ? t[k] : -t[k];
    if (cy(i)) jy += cy(i) > 0 ? t[k] : -t[k];
    if (cz(i)) jz += cz(i) > 0 ? t[k] : -t[k];
  }
  const float inv = 1.0f / (1.0f + drho);
  const float ux = jx * inv, uy = jy * inv, uz = jz * inv;
  const float B = drho - 1.5f * (jx * ux + jy * uy + jz * uz);
  float E[9];  // even part of feq / w
  auto even = [&](auto kk) {
    constexpr int k = decltype(kk)::value;
    E[k] = B + 4.5f * along<k>(jx, jy, jz) * along<k>(ux, uy, uz);
  };
  each_pair(even);
  float omega = c.omega;
  if (KIND == KIND_SMAG) {
    float pxx = 0.f, pyy = 0.f, pzz = 0.f, pxy = 0.f, pxz = 0.f, pyz = 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const int i = pos_dir(k);
      const float n = s[k] - 2.0f * wf(i) * E[k];
      if (cx(i)) pxx += n;
      if (cy(i)) pyy += n;
      if (cz(i)) pzz += n;
      if (cx(i) && cy(i)) pxy += cx(i) * cy(i) > 0 ? n : -n;
      if (cx(i) && cz(i)) pxz += cx(i) * cz(i) > 0 ? n : -n;
      if (cy(i) && cz(i)) pyz += cy(i) * cz(i) > 0 ? n : -n;
    }
    const float pp =
        pxx * pxx + pyy * pyy + pzz * pzz + 2.0f * (pxy * pxy + pxz * pxz + pyz * pyz);
    omega = smagorinsky_omega(pp, inv, c.tau, c.tau0_sq, c.smag_c18);
  }
  const float j3x = 3.0f * jx, j3y = 3.0f * jy, j3z = 3.0f * jz;
  const float sx = 2.0f * ux + Fx * inv, sy = 2.0f * uy + Fy * inv, sz = 2.0f * uz + Fz * inv;
  const float Fs = 1.5f * (Fx * sx + Fy * sy + Fz * sz);
  d[0] = fmaf(omega, wf(0) * B - d[0], d[0]) - wf(0) * Fs;
  auto relax = [&](auto kk) {
    constexpr int k = decltype(kk)::value, i = pos_dir(k), o = opposite(i);
    const float cF = along<k>(Fx, Fy, Fz), cs = along<k>(sx, sy, sz);
    const float q = along<k>(j3x, j3y, j3z);
    const float fe = 4.5f * cF * cs - Fs, fo = 3.0f * cF;
    d[i] = fmaf(wf(i), fe + fo, fmaf(omega, wf(i) * (E[k] + q) - d[i], d[i]));
    d[o] = fmaf(wf(i), fe - fo, fmaf(omega, wf(i) * (E[k] - q) - d[o], d[o]));
  };
  each_pair(relax);
  const float usq = ux * ux + uy * uy + uz * uz;
  return !(usq < UNSTABLE_USQ);
}

// I: type of the node offsets within a lattice.  32-bit ones leave the plane
// bases to the uniform registers.
template <int KIND, class I>
__global__ void __launch_bounds__(NT) k3_step(const float *__restrict__ in, float *__restrict__ out,
                                              Grid3 g, Collide3 c, int *flag) {
  umma::griddep_wait();  // launched as a dependent of the previous step
  umma::griddep_launch_dependents();
  Pos p;
  if (!node_pos(g, p)) return;
  const size_t vol = g.volume();
  const float *gb = in + (size_t)p.b * Q * vol;
  // sources x - c_x, and rows (z - c_z, y - c_y), at 1 + c
  const I nx = (I)g.nx;
  const I xs[3] = {(I)(p.x == g.nx - 1 ? 0 : p.x + 1), (I)p.x, (I)(p.x == 0 ? g.nx - 1 : p.x - 1)};
  const int ys[3] = {p.y == g.ny - 1 ? 0 : p.y + 1, p.y, p.y == 0 ? g.ny - 1 : p.y - 1};
  const int zs[3] = {p.z == g.nz - 1 ? 0 : p.z + 1, p.z, p.z == 0 ? g.nz - 1 : p.z - 1};
  float d[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const I row = ((I)zs[1 + cz(i)] * (I)g.ny + (I)ys[1 + cy(i)]) * nx;  // uniform
    d[i] = __ldg(gb + (size_t)i * vol + (row + xs[1 + cx(i)]));
  }
  float Fx, Fy, Fz;
  node_force(c, p, Fx, Fy, Fz);
  flag_bad(collide_pairs<KIND>(d, c, Fx, Fy, Fz), flag);
  float *o = out + (size_t)p.b * Q * vol;
  const I n = ((I)p.z * (I)g.ny + (I)p.y) * nx + (I)p.x;
#pragma unroll
  for (int i = 0; i < Q; ++i) (o + (size_t)i * vol)[n] = d[i];
}

// state_i(x) = f_i(x + c_i) - w_i (anti-streaming into the pull representation)
__global__ void k3_set_state(const float *__restrict__ f, float *__restrict__ st, Grid3 g) {
  Pos p;
  if (!node_pos(g, p)) return;
  const size_t vol = g.volume(), base = (size_t)p.b * Q * vol;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int xs = wrapi(p.x + cx(i), g.nx), ys = wrapi(p.y + cy(i), g.ny),
              zs = wrapi(p.z + cz(i), g.nz);
    st[base + (size_t)i * vol + at(g, p)] =
        f[base + (size_t)i * vol + ((size_t)zs * g.ny + ys) * g.nx + xs] - wf(i);
  }
}

// f_i(x) = state_i(x - c_i) + w_i
__global__ void k3_get_state(const float *__restrict__ st, float *__restrict__ f, Grid3 g) {
  Pos p;
  if (!node_pos(g, p)) return;
  float d[Q];
  pull(st, g, p, d);
  const size_t vol = g.volume(), base = (size_t)p.b * Q * vol;
#pragma unroll
  for (int i = 0; i < Q; ++i) f[base + (size_t)i * vol + at(g, p)] = d[i] + wf(i);
}

// feq(rho, u) at x becomes the pre-collision state: written to x - c_i.
__global__ void k3_init_equilibrium(const float *__restrict__ rho, const float *__restrict__ u,
                                    float *__restrict__ st, Grid3 g) {
  Pos p;
  if (!node_pos(g, p)) return;
  const size_t vol = g.volume(), base = (size_t)p.b * Q * vol;
  const size_t n = at(g, p);
  Moments m;
  m.rho = rho[(size_t)p.b * vol + n];
  m.drho = m.rho - 1.0f;
  m.ux = u[((size_t)p.b * 3 + 0) * vol + n];
  m.uy = u[((size_t)p.b * 3 + 1) * vol + n];
  m.uz = u[((size_t)p.b * 3 + 2) * vol + n];
  float deq[Q];
  shifted_feq(m, deq);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int xs = wrapi(p.x - cx(i), g.nx), ys = wrapi(p.y - cy(i), g.ny),
              zs = wrapi(p.z - cz(i), g.nz);
    st[base + (size_t)i * vol + ((size_t)zs * g.ny + ys) * g.nx + xs] = deq[i];
  }
}

// rho [b][z][y][x] and u [b][3][z][y][x] of the pre-collision populations
__global__ void k3_moments(const float *__restrict__ st, float *rho, float *u, Grid3 g) {
  Pos p;
  if (!node_pos(g, p)) return;
  float d[Q];
  pull(st, g, p, d);
  const Moments m = node_moments(d);
  const size_t vol = g.volume(), n = at(g, p);
  if (rho) rho[(size_t)p.b * vol + n] = m.rho;
  if (u) {
    u[((size_t)p.b * 3 + 0) * vol + n] = m.ux;
    u[((size_t)p.b * 3 + 1) * vol + n] = m.uy;
    u[((size_t)p.b * 3 + 2) * vol + n] = m.uz;
  }
}

dim3 node_grid(const Grid3 &g) { return dim3((g.nx + NT - 1) / NT, g.ny, g.nz * g.batch); }

}  // namespace

// Programmatic dependent launch: the kernel waits for the previous kernel on
// the stream before its first global access, which hides the launch gap.
cudaError_t launch_step(const Grid3 &g, const float *in, float *out, const Collide3 &c, int kind,
                        int *flag, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = node_grid(g);
  cfg.blockDim = dim3(NT);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (g.volume() >= 1u << 31) {
    auto kern = kind == KIND_SMAG ? k3_step<KIND_SMAG, size_t> : k3_step<KIND_BGK, size_t>;
    return cudaLaunchKernelEx(&cfg, kern, in, out, g, c, flag);
  }
  auto kern = kind == KIND_SMAG ? k3_step<KIND_SMAG, unsigned> : k3_step<KIND_BGK, unsigned>;
  return cudaLaunchKernelEx(&cfg, kern, in, out, g, c, flag);
}

cudaError_t launch_set_state(const Grid3 &g, const float *f_pre, float *state, cudaStream_t s) {
  k3_set_state<<<node_grid(g), NT, 0, s>>>(f_pre, state, g);
  return cudaGetLastError();
}

cudaError_t launch_get_state(const Grid3 &g, const float *state, float *f_pre, cudaStream_t s) {
  k3_get_state<<<node_grid(g), NT, 0, s>>>(state, f_pre, g);
  return cudaGetLastError();
}

cudaError_t launch_init_equilibrium(const Grid3 &g, const float *rho, const float *u,
                                    float *state, cudaStream_t s) {
  k3_init_equilibrium<<<node_grid(g), NT, 0, s>>>(rho, u, state, g);
  return cudaGetLastError();
}

cudaError_t launch_moments(const Grid3 &g, const float *state, float *rho, float *u,
                           cudaStream_t s) {
  k3_moments<<<node_grid(g), NT, 0, s>>>(state, rho, u, g);
  return cudaGetLastError();
}

}  // namespace d3
}  // namespace lbm
