// d3q19_step.cu -- the paper's 3D setting on the CUDA cores: the fused D3Q19
// pull-stream + BGK / Smagorinsky-BGK step with the paper's three-component sine
// forcing (EDM, Eq. S5), and the data-movement kernels around it.
//
// Step kernels: one thread per node along x; each pulls f_i(x) = g_i(x - c_i)
// (periodic) from the previous buffer, collides and stores at x.  Algorithmic
// traffic 76 B read + 76 B written per node.
#include "d3q19.cuh"
#include "kernels3d.h"
#include "umma.cuh"

namespace lbm {
namespace d3 {
namespace {

constexpr int NT = 128;
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

template <int KIND>
__global__ void __launch_bounds__(NT) k3_step(const float *__restrict__ in, float *__restrict__ out,
                                              Grid3 g, Collide3 c, int *flag) {
  umma::griddep_wait();  // launched as a dependent of the previous step
  umma::griddep_launch_dependents();
  Pos p;
  if (!node_pos(g, p)) return;
  float d[Q], deq[Q];
  pull(in, g, p, d);
  const Moments m = node_moments(d);
  shifted_feq(m, deq);
  const float om = KIND == KIND_SMAG ? smag_omega(d, deq, m.inv_rho, c.tau0_sq, c.tau, c.smag_c18)
                                     : c.omega;
#pragma unroll
  for (int i = 0; i < Q; ++i) d[i] += om * (deq[i] - d[i]);
  float Fx, Fy, Fz;
  node_force(c, p, Fx, Fy, Fz);
  add_edm_force(m, Fx, Fy, Fz, d);
  flag_bad(is_unstable(m), flag);
  const size_t vol = g.volume();
  float *o = out + (size_t)p.b * Q * vol + at(g, p);
#pragma unroll
  for (int i = 0; i < Q; ++i) o[(size_t)i * vol] = d[i];
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
  if (kind == KIND_SMAG) return cudaLaunchKernelEx(&cfg, k3_step<KIND_SMAG>, in, out, g, c, flag);
  return cudaLaunchKernelEx(&cfg, k3_step<KIND_BGK>, in, out, g, c, flag);
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
