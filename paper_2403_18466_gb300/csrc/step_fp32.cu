// step_fp32.cu -- HBM-bound FP32 kernels: the fused pull-stream + BGK /
// Smagorinsky-BGK step (+ EDM forcing), and the data-movement kernels
// around it (state in/out, equilibrium init, moments, box and subsampling
// filters, full-field and node-subset losses, push/pull of a field).
//
// Step kernel (Eq. S2 with the stream/collide split of the Methods section):
// each node pulls f_i(x) = g_i(x - c_i) from the previous buffer, collides
// (Eq. S3, or SI section 1 for Smagorinsky), adds the EDM force (Eq. S5) and
// stores into the next buffer at x.  Algorithmic traffic: 36 B read + 36 B
// written per node (FP32 D2Q9).
//
// Several steps of one call run as one launch (k_steps_tile; k_steps_small on
// small lattices).  Single steps:
// nx % 4 == 0: one thread owns 4 consecutive nodes of a row.
// Every plane row is read with aligned 128-bit loads; the one value that a
// shifted plane (c_x = +-1) needs from the neighbouring 4-node group comes
// from the adjacent lane by a warp shuffle, and only the warp's edge lanes
// (and the periodic wrap) issue an extra scalar load.  Stores are aligned
// 128-bit.  Other widths take a one-node-per-thread kernel.
#include <algorithm>
#include <cmath>

#include "approx.cuh"
#include "kernels.h"
#include "lattice.cuh"
#include "umma.cuh"

namespace lbm {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int VEC_THREADS = 128;  // 512 nodes of one row per block
constexpr int SCALAR_THREADS = 128;

enum { KIND_BGK = 0, KIND_SMAG = 1 };

__device__ __forceinline__ float smag_omega(float pp, float inv_rho, const CollideParams &p) {
  return smagorinsky_omega(pp, inv_rho, p.tau, p.tau0_sq, p.smag_c18);
}
__device__ __forceinline__ float2 smag_omega(float2 pp, float2 inv_rho, const CollideParams &p) {
  return make_float2(smag_omega(pp.x, inv_rho.x, p), smag_omega(pp.y, inv_rho.y, p));
}

__device__ __forceinline__ bool unstable(const MomentsT<float> &m, bool, bool) {
  return is_unstable(m);
}
__device__ __forceinline__ bool unstable(const MomentsT<float2> &m, bool x, bool y) {
  return is_unstable(m, x, y);
}

// Collide one node (float) or two (float2: packed f32x2, half the issue slots)
// in place (shifted representation), add the force.  Every operation is
// rounded explicitly, so both forms, and every kernel that uses them, give the
// same bits.  Returns true if a node is unstable (|u| >= 0.4 or not finite;
// act_x, act_y: which of two nodes count).
//
// BGK: the operations of the learned kernels, which reduce to it bit for bit.
template <class T>
__device__ __forceinline__ bool collide_bgk(T d[Q], const CollideParams &p, T fx, bool act_x,
                                            bool act_y) {
  const MomentsT<T> m = node_moments(d);
  const bool bad = unstable(m, act_x, act_y);
  T deq[Q];
  shifted_feq(m, deq);
#pragma unroll
  for (int i = 0; i < Q; ++i) d[i] = bgk_relax(d[i], deq[i], v_c<T>(p.omega));
  add_edm_force_x(m, fx, d);  // fx = 0 without forcing
  return bad;
}

// Smagorinsky, on the even and odd parts s = f_i + f_opp, t = f_i - f_opp of the
// opposite pairs (1, 3), (2, 4), (5, 7), (6, 8): feq's even part is w E with
// E = drho - 1.5 j.u + 4.5 (c.j)(c.u) and its odd part 3 w c.j, so a pair shares E,
// and Pi^neq_ab = sum c_a c_b (f - feq) needs the even parts alone: about two thirds
// of the FP32 operations of the sums direction by direction.
template <class T>
__device__ __forceinline__ bool collide_smag(T d[Q], const CollideParams &p, T fx, bool act_x,
                                             bool act_y) {
  const T sx = v_add(d[1], d[3]), sy = v_add(d[2], d[4]), sd = v_add(d[5], d[7]),
          sa = v_add(d[6], d[8]);
  const T td = v_sub(d[5], d[7]), ta = v_sub(d[6], d[8]);
  MomentsT<T> m;
  m.drho = v_add(d[0], v_add(v_add(sx, sy), v_add(sd, sa)));
  const T jx = v_add(v_sub(d[1], d[3]), v_sub(td, ta));
  const T jy = v_add(v_sub(d[2], d[4]), v_add(td, ta));
  m.rho = v_add(v_c<T>(1.0f), m.drho);
  m.inv_rho = v_rcp(m.rho);
  m.ux = v_mul(jx, m.inv_rho);
  m.uy = v_mul(jy, m.inv_rho);
  const bool bad = unstable(m, act_x, act_y);
  const T xx = v_mul(jx, m.ux), yy = v_mul(jy, m.uy), c45 = v_c<T>(4.5f);
  const T B = v_fma(v_c<T>(-1.5f), v_add(xx, yy), m.drho);
  const T jd = v_add(jx, jy), ja = v_sub(jy, jx);
  const T Ex = v_fma(c45, xx, B), Ey = v_fma(c45, yy, B);
  const T Ed = v_fma(c45, v_mul(jd, v_add(m.ux, m.uy)), B);
  const T Ea = v_fma(c45, v_mul(ja, v_sub(m.uy, m.ux)), B);
  // tau_eff in closed form (SI sec. 1)
  const T w1 = v_c<T>(wf(1)), w5 = v_c<T>(wf(5));
  const T m1 = v_c<T>(-2.0f * wf(1)), m5 = v_c<T>(-2.0f * wf(5));
  const T nd = v_fma(m5, Ed, sd), na = v_fma(m5, Ea, sa), diag = v_add(nd, na);
  const T pxx = v_add(v_fma(m1, Ex, sx), diag), pyy = v_add(v_fma(m1, Ey, sy), diag);
  const T pxy = v_sub(nd, na);
  const T pp = v_fma(pyy, pyy, v_fma(v_mul(v_c<T>(2.0f), pxy), pxy, v_mul(pxx, pxx)));
  const T omega = smag_omega(pp, m.inv_rho, p);
  // f + omega (feq - f), feq = w (E +- 3 c.j)
  const T three = v_c<T>(3.0f);
  auto relax = [&](T &a, T &b, T w, T E, T cj) {
    a = v_fma(omega, v_sub(v_mul(w, v_fma(three, cj, E)), a), a);
    b = v_fma(omega, v_sub(v_mul(w, v_fma(v_c<T>(-3.0f), cj, E)), b), b);
  };
  d[0] = v_fma(omega, v_sub(v_mul(v_c<T>(wf(0)), B), d[0]), d[0]);
  relax(d[1], d[3], w1, Ex, jx);
  relax(d[2], d[4], w1, Ey, jy);
  relax(d[5], d[7], w5, Ed, jd);
  relax(d[6], d[8], w5, Ea, ja);
  add_edm_force_x(m, fx, d);  // fx = 0 without forcing
  return bad;
}

template <int KIND, class T>
__device__ __forceinline__ bool collide_node(T d[Q], const CollideParams &p, T fx,
                                             bool act_x = true, bool act_y = true) {
  return KIND == KIND_SMAG ? collide_smag(d, p, fx, act_x, act_y)
                           : collide_bgk(d, p, fx, act_x, act_y);
}

__device__ __forceinline__ float4 ldg4(const float *p) {
  return __ldg(reinterpret_cast<const float4 *>(p));
}

// Values g(x0 - CXI .. x0 + 3 - CXI) of one plane row, for the 4-node group
// starting at x0 (x0 % 4 == 0).  All lanes must call it (warp shuffles).
template <int CXI>
__device__ __forceinline__ void pull4(const float *__restrict__ row, int x0, int nx, int lane,
                                      bool active, float v[4]) {
  const float4 a = active ? ldg4(row + x0) : make_float4(0.f, 0.f, 0.f, 0.f);
  if (CXI == 0) {
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  } else if (CXI == 1) {  // needs x0 - 1 .. x0 + 2
    float prev = __shfl_up_sync(FULL, a.w, 1);
    if (active && lane == 0) prev = __ldg(row + (x0 == 0 ? nx - 1 : x0 - 1));
    v[0] = prev; v[1] = a.x; v[2] = a.y; v[3] = a.z;
  } else {  // CXI == -1: needs x0 + 1 .. x0 + 4
    float next = __shfl_down_sync(FULL, a.x, 1);
    if (active && (lane == 31 || x0 + 4 >= nx)) next = __ldg(row + (x0 + 4 >= nx ? x0 + 4 - nx : x0 + 4));
    v[0] = a.y; v[1] = a.z; v[2] = a.w; v[3] = next;
  }
}

template <int I>
__device__ __forceinline__ void pull_plane4(const float *__restrict__ gb, size_t plane, int nx,
                                            int y, int ym, int yp, int x0, int lane, bool active,
                                            float v[Q][4]) {
  const int ys = cy(I) == 0 ? y : (cy(I) == 1 ? ym : yp);  // source row y - c_iy
  pull4<cx(I)>(gb + I * plane + (size_t)ys * nx, x0, nx, lane, active, v[I]);
}

template <int KIND>
__global__ void __launch_bounds__(VEC_THREADS)
    k_step_vec(const float *__restrict__ in, float *__restrict__ out, int nx, int ny,
               CollideParams p, int *flag) {
  umma::griddep_wait();  // launched as a dependent of the previous step
  umma::griddep_launch_dependents();
  const int lane = threadIdx.x & 31;
  const int x0 = (blockIdx.x * VEC_THREADS + threadIdx.x) * 4;
  const int y = blockIdx.y;
  const size_t plane = (size_t)nx * ny;
  const float *gb = in + (size_t)blockIdx.z * Q * plane;
  float *ob = out + (size_t)blockIdx.z * Q * plane;
  const bool active = x0 < nx;
  const int ym = y == 0 ? ny - 1 : y - 1;
  const int yp = y == ny - 1 ? 0 : y + 1;
  float v[Q][4];
  pull_plane4<0>(gb, plane, nx, y, ym, yp, x0, lane, active, v);
  pull_plane4<1>(gb, plane, nx, y, ym, yp, x0, lane, active, v);
  pull_plane4<2>(gb, plane, nx, y, ym, yp, x0, lane, active, v);
  pull_plane4<3>(gb, plane, nx, y, ym, yp, x0, lane, active, v);
  pull_plane4<4>(gb, plane, nx, y, ym, yp, x0, lane, active, v);
  pull_plane4<5>(gb, plane, nx, y, ym, yp, x0, lane, active, v);
  pull_plane4<6>(gb, plane, nx, y, ym, yp, x0, lane, active, v);
  pull_plane4<7>(gb, plane, nx, y, ym, yp, x0, lane, active, v);
  pull_plane4<8>(gb, plane, nx, y, ym, yp, x0, lane, active, v);
  const float fx = p.force ? __ldg(p.force + y) : 0.0f;
  bool bad = false;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float d[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) d[i] = v[i][k];
    bad |= collide_node<KIND>(d, p, fx);
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i][k] = d[i];
  }
  flag_unstable(bad && active, flag);
  if (!active) return;
#pragma unroll
  for (int i = 0; i < Q; ++i)
    *reinterpret_cast<float4 *>(ob + i * plane + (size_t)y * nx + x0) =
        make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
}

// Gather the 9 pulled values of node (x, y): d_i = g_i(x - c_i).
__device__ __forceinline__ void pull_node(const float *__restrict__ gb, size_t plane, int nx,
                                          int ny, int x, int y, float d[Q]) {
  const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
  const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int xs = cx(i) == 0 ? x : (cx(i) == 1 ? xm : xp);
    const int ys = cy(i) == 0 ? y : (cy(i) == 1 ? ym : yp);
    d[i] = __ldg(gb + i * plane + (size_t)ys * nx + xs);
  }
}

template <int KIND>
__global__ void __launch_bounds__(SCALAR_THREADS)
    k_step_scalar(const float *__restrict__ in, float *__restrict__ out, int nx, int ny,
                  CollideParams p, int *flag) {
  umma::griddep_wait();  // launched as a dependent of the previous step
  umma::griddep_launch_dependents();
  const int x = blockIdx.x * SCALAR_THREADS + threadIdx.x;
  const int y = blockIdx.y;
  if (x >= nx) return;
  const size_t plane = (size_t)nx * ny;
  const float *gb = in + (size_t)blockIdx.z * Q * plane;
  float *ob = out + (size_t)blockIdx.z * Q * plane;
  float d[Q];
  pull_node(gb, plane, nx, ny, x, y, d);
  const bool bad = collide_node<KIND>(d, p, p.force ? __ldg(p.force + y) : 0.0f);
  flag_unstable(bad, flag);
#pragma unroll
  for (int i = 0; i < Q; ++i) ob[i * plane + (size_t)y * nx + x] = d[i];
}

// Several steps in one pass over memory: a block advances a tile by t steps
// (t <= MT_MOST), the first on a region of MT_X x MT_Y nodes and each later one
// on a ring less, and stores the (MT_X - 2 (t - 1)) x (MT_Y - 2 (t - 1)) nodes
// that are then complete, so the state crosses HBM (or L2) once per t steps.
// A thread owns MT_PP pairs of adjacent rows of one column: the two nodes of a
// pair run in packed f32x2 arithmetic, and their 18 populations are plain
// 32-bit loads (a warp reads 32 adjacent columns of a row), with no shuffles
// and no moves to form the pairs.  Between steps the post-collision
// populations are in shared memory, replaced in place.
// What bounds it: the FP32 pipe and instruction issue, no longer HBM (55 % and
// 64 % busy at 1024^2 Smagorinsky before its collision took the form of even and
// odd parts); t = 3 on a 64 x 16 region recomputes 21 % of the nodes.  Measured (GB300, us per
// step, BGK / Smagorinsky, one step per launch before):
//   256^2   3.2 / 3.6 -> 1.6 / 1.7       512^2   4.6 / 5.0 -> 2.8 / 3.2
//   1024^2 10.0 / 10.6 -> 8.4 / 9.2     2048^2  49.5 / 51.8 -> 30.3 / 33.1
//   4096^2  185 / 189 -> 115 / 126      1001^2  11.0 / 12.0 -> 7.9 / 8.6
// (Smagorinsky direction by direction: 1.9, 3.5, 10.4, 36.6, 140, 9.6.)
// t = 2 or 4, 32- or 24-row regions and other block sizes were within 15 % or
// slower; four nodes per thread with 128-bit loads and shuffles (t = 2) reached
// 41 us at 2048^2, the same with the next tile's cp.async copies in flight 44.
constexpr int MT_X = 64, MT_THREADS = 256, MT_PR = MT_THREADS / MT_X;
constexpr int MT_PP = 2;               // pairs of rows per thread
constexpr int MT_Y = 2 * MT_PR * MT_PP;  // rows of the region
constexpr int MT_MOST = 3;

template <int KIND>
__global__ void __launch_bounds__(MT_THREADS, 3)
    k_steps_tile(const float *__restrict__ in, float *__restrict__ out, int nx, int ny, int t,
                 CollideParams p, int *flag) {
  constexpr int RY = MT_Y, PP = MT_PP;
  extern __shared__ float tile[];  // [Q][RY][MT_X]
  umma::griddep_wait();  // launched as a dependent of the previous step
  umma::griddep_launch_dependents();
  const int lx = threadIdx.x % MT_X, pr = threadIdx.x / MT_X;
  const int X0 = (int)blockIdx.x * (MT_X - 2 * (t - 1)) - (t - 1);
  const int Y0 = (int)blockIdx.y * (RY - 2 * (t - 1)) - (t - 1);
  const size_t plane = (size_t)nx * ny;
  auto wrap = [](int a, int n) { return a < 0 ? (a % n + n) % n : (a >= n ? a % n : a); };
  bool bad = false;
  float2 d[PP][Q];
  float2 fx[PP];
  {
    // step 1, from global memory
    const float *gb = in + (size_t)blockIdx.z * Q * plane;
    const uint32_t x = wrap(X0 + lx, nx), X = nx;
    // x - c_x at 1 + c_x
    const uint32_t xs[3] = {x == X - 1 ? 0 : x + 1, x, x == 0 ? X - 1 : x - 1};
#pragma unroll
    for (int j = 0; j < PP; ++j) {
      const int y0 = wrap(Y0 + 2 * (pr + MT_PR * j), ny);
      const int y1 = y0 == ny - 1 ? 0 : y0 + 1;
      const int ym = y0 == 0 ? ny - 1 : y0 - 1, yp = y1 == ny - 1 ? 0 : y1 + 1;
      // source rows of the two nodes, y - c_y at 1 + c_y
      const uint32_t r0[3] = {y1 * X, y0 * X, ym * X}, r1[3] = {yp * X, y1 * X, y0 * X};
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const float *pl = gb + i * plane;
        d[j][i] = make_float2(__ldg(pl + (r0[1 + cy(i)] + xs[1 + cx(i)])),
                              __ldg(pl + (r1[1 + cy(i)] + xs[1 + cx(i)])));
      }
      fx[j] = p.force ? make_float2(__ldg(p.force + y0), __ldg(p.force + y1))
                      : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int j = 0; j < PP; ++j) bad |= collide_node<KIND>(d[j], p, fx[j], true, true);
  }
#pragma unroll 1
  for (int s = 1; s < t; ++s) {
    if (s > 1) __syncthreads();  // the previous state is read
#pragma unroll
    for (int j = 0; j < PP; ++j) {
      float *o = tile + 2 * (pr + MT_PR * j) * MT_X + lx;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        o[i * RY * MT_X] = d[j][i].x;
        o[i * RY * MT_X + MT_X] = d[j][i].y;
      }
    }
    __syncthreads();
    // nodes at least s from the region's edge; the other node of a pair that
    // straddles the limit reads a clamped row and is not used
    if (lx >= s && lx < MT_X - s) {
#pragma unroll
      for (int j = 0; j < PP; ++j) {
        const int r = 2 * (pr + MT_PR * j);
        if (r + 1 < s || r >= RY - s) continue;
        const int rm = r == 0 ? 0 : r - 1, rp = r + 2 == RY ? r + 1 : r + 2;
        const int a[3] = {r + 1, r, rm}, b[3] = {rp, r + 1, r};
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          const float *pl = tile + i * RY * MT_X + lx - cx(i);
          d[j][i] = make_float2(pl[a[1 + cy(i)] * MT_X], pl[b[1 + cy(i)] * MT_X]);
        }
        bad |= collide_node<KIND>(d[j], p, fx[j], r >= s, r + 1 < RY - s);
      }
    }
  }
  flag_unstable(bad, flag);
  const int e = t - 1, x = X0 + lx;
  if (lx < e || lx >= MT_X - e || x >= nx) return;
  float *ob = out + (size_t)blockIdx.z * Q * plane;
#pragma unroll
  for (int j = 0; j < PP; ++j) {
    const int r = 2 * (pr + MT_PR * j), y = Y0 + r;
    const uint32_t at = (uint32_t)y * (uint32_t)nx + (uint32_t)x;
    if (r >= e && r < RY - e && y < ny)
#pragma unroll
      for (int i = 0; i < Q; ++i) (ob + i * plane)[at] = d[j][i].x;
    if (r + 1 >= e && r + 1 < RY - e && y + 1 < ny)
#pragma unroll
      for (int i = 0; i < Q; ++i) (ob + i * plane)[at + (uint32_t)nx] = d[j][i].y;
  }
}

// Several steps in one launch for small lattices, where the launches are the
// cost (64^2 BGK: 2.9 us per step with one step per launch, 0.66 with 8): a
// block advances a tile of ts x ts nodes by t steps, the first on the tile and
// the t - 1 nodes around it (one node per thread), each later one on a ring
// less, between two shared-memory buffers.
constexpr int MS_SIDE = 22;               // ts + 2 (t - 1) at most
constexpr int MS_NODES = MS_SIDE * MS_SIDE;
constexpr int MS_THREADS = 512;
static_assert(MS_NODES <= MS_THREADS, "one node per thread");

template <int KIND>
__global__ void __launch_bounds__(MS_THREADS, 2)
    k_steps_small(const float *__restrict__ in, float *__restrict__ out, int nx, int ny, int ts,
                  int t, CollideParams p, int *flag) {
  extern __shared__ float buf[];  // [2][Q][MS_NODES]
  umma::griddep_wait();           // launched as a dependent of the previous step
  umma::griddep_launch_dependents();
  const int side = ts + 2 * (t - 1);
  const int ly = threadIdx.x / side, lx = threadIdx.x - ly * side;
  const size_t plane = (size_t)nx * ny;
  const bool node = ly < side;
  int x = 0, y = 0;
  if (node) {
    x = ((int)blockIdx.x * ts - (t - 1) + lx) % nx;
    y = ((int)blockIdx.y * ts - (t - 1) + ly) % ny;
    x = x < 0 ? x + nx : x;
    y = y < 0 ? y + ny : y;
  }
  const float fx = p.force && node ? __ldg(p.force + y) : 0.0f;
  // this node takes part in the first `steps` steps
  const int edge = min(min(lx, side - 1 - lx), min(ly, side - 1 - ly));
  const int steps = node ? min(edge + 1, t) : 0;
  float d[Q];
  bool bad = false;
  if (node) {
    pull_node(in + (size_t)blockIdx.z * Q * plane, plane, nx, ny, x, y, d);
    bad = collide_node<KIND>(d, p, fx);
  }
  for (int s = 1; s < t; ++s) {
    float *b = buf + (s & 1) * (Q * MS_NODES);
    if (s <= steps)
#pragma unroll
      for (int i = 0; i < Q; ++i) b[i * MS_NODES + threadIdx.x] = d[i];
    __syncthreads();
    if (s < steps) {
#pragma unroll
      for (int i = 0; i < Q; ++i) d[i] = b[i * MS_NODES + (int)threadIdx.x - cy(i) * side - cx(i)];
      bad |= collide_node<KIND>(d, p, fx);
    }
  }
  flag_unstable(bad, flag);
  const int gx = blockIdx.x * ts + lx - (t - 1), gy = blockIdx.y * ts + ly - (t - 1);
  if (steps == t && gx < nx && gy < ny) {
    float *ob = out + (size_t)blockIdx.z * Q * plane + (size_t)gy * nx + gx;
#pragma unroll
    for (int i = 0; i < Q; ++i) ob[i * plane] = d[i];
  }
}

// Programmatic dependent launch: the kernel waits for the previous kernel on
// the stream before its first global access, so its CTAs may be scheduled
// while that kernel's last CTAs finish (it hides the launch gap between steps).
template <int KIND>
cudaError_t launch_steps(const Grid &g, const float *in, float *out, const CollideParams &p, int t,
                         int *flag, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const StepPlan plan = step_plan(g);
  if (t > 1 && plan.tile > 0) {
    constexpr size_t smem = 2 * Q * MS_NODES * sizeof(float);
    static_assert(smem <= 48 * 1024, "what a launch may take without asking");
    cfg.gridDim = dim3((g.nx + plan.tile - 1) / plan.tile, (g.ny + plan.tile - 1) / plan.tile,
                       g.batch);
    cfg.blockDim = dim3(MS_THREADS);
    cfg.dynamicSmemBytes = smem;
    return cudaLaunchKernelEx(&cfg, k_steps_small<KIND>, in, out, g.nx, g.ny, plan.tile, t, p, flag);
  }
  if (t > 1) {
    constexpr size_t smem = Q * MT_Y * MT_X * sizeof(float);
    static_assert(smem <= 48 * 1024, "what a launch may take without asking");
    const int tw = MT_X - 2 * (t - 1), th = MT_Y - 2 * (t - 1);
    cfg.gridDim = dim3((g.nx + tw - 1) / tw, (g.ny + th - 1) / th, g.batch);
    cfg.blockDim = dim3(MT_THREADS);
    cfg.dynamicSmemBytes = smem;
    return cudaLaunchKernelEx(&cfg, k_steps_tile<KIND>, in, out, g.nx, g.ny, t, p, flag);
  }
  const bool vec = g.nx % 4 == 0;
  cfg.gridDim = vec ? dim3((g.nx / 4 + VEC_THREADS - 1) / VEC_THREADS, g.ny, g.batch)
                    : dim3((g.nx + SCALAR_THREADS - 1) / SCALAR_THREADS, g.ny, g.batch);
  cfg.blockDim = dim3(vec ? VEC_THREADS : SCALAR_THREADS);
  if (vec) return cudaLaunchKernelEx(&cfg, k_step_vec<KIND>, in, out, g.nx, g.ny, p, flag);
  return cudaLaunchKernelEx(&cfg, k_step_scalar<KIND>, in, out, g.nx, g.ny, p, flag);
}

// ---------------------------------------------------------------------------
// Node-parallel helpers: one thread per node, grid (ceil(nx/128), ny, batch).
// ---------------------------------------------------------------------------
constexpr int NT = 128;

__device__ __forceinline__ bool node_index(int nx, int &x, int &y, int &b) {
  x = blockIdx.x * NT + threadIdx.x;
  y = blockIdx.y;
  b = blockIdx.z;
  return x < nx;
}

dim3 node_grid(const Grid &g) { return dim3((g.nx + NT - 1) / NT, g.ny, g.batch); }

// state_i(x) = f_i(x + c_i) - w_i  (anti-streaming, SI section 2 step 4)
__global__ void k_set_state(const float *__restrict__ f, float *__restrict__ st, int nx, int ny) {
  int x, y, b;
  if (!node_index(nx, x, y, b)) return;
  const size_t plane = (size_t)nx * ny, base = (size_t)b * Q * plane;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int xs = wrap_index(x + cx(i), nx), ys = wrap_index(y + cy(i), ny);
    st[base + i * plane + (size_t)y * nx + x] = f[base + i * plane + (size_t)ys * nx + xs] - wf(i);
  }
}

// f_i(x) = state_i(x - c_i) + w_i
__global__ void k_get_state(const float *__restrict__ st, float *__restrict__ f, int nx, int ny) {
  int x, y, b;
  if (!node_index(nx, x, y, b)) return;
  const size_t plane = (size_t)nx * ny, base = (size_t)b * Q * plane;
  float d[Q];
  pull_node(st + base, plane, nx, ny, x, y, d);
#pragma unroll
  for (int i = 0; i < Q; ++i) f[base + i * plane + (size_t)y * nx + x] = d[i] + wf(i);
}

// feq(rho, u) at node x becomes the pre-collision state: written to x - c_i.
__global__ void k_init_equilibrium(const float *__restrict__ rho, const float *__restrict__ ux,
                                   const float *__restrict__ uy, float *__restrict__ st, int nx,
                                   int ny) {
  int x, y, b;
  if (!node_index(nx, x, y, b)) return;
  const size_t plane = (size_t)nx * ny, base = (size_t)b * Q * plane;
  const size_t n = (size_t)b * plane + (size_t)y * nx + x;
  Moments m;
  m.rho = rho[n];
  m.drho = m.rho - 1.0f;
  m.ux = ux[n];
  m.uy = uy[n];
  float deq[Q];
  shifted_feq(m, deq);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int xs = wrap_index(x - cx(i), nx), ys = wrap_index(y - cy(i), ny);
    st[base + i * plane + (size_t)ys * nx + xs] = deq[i];
  }
}

__global__ void k_moments(const float *__restrict__ st, float *rho, float *ux, float *uy, int nx,
                          int ny) {
  int x, y, b;
  if (!node_index(nx, x, y, b)) return;
  const size_t plane = (size_t)nx * ny;
  float d[Q];
  pull_node(st + (size_t)b * Q * plane, plane, nx, ny, x, y, d);
  const Moments m = node_moments(d);
  const size_t n = (size_t)b * plane + (size_t)y * nx + x;
  if (rho) rho[n] = m.rho;
  if (ux) ux[n] = m.ux;
  if (uy) uy[n] = m.uy;
}

// A sum of floats as three: h + l + m, every rounding error of h caught in l and
// every one of l in m (Knuth's two-sum), so more than the 53 bits of a double.
struct Sum3 {
  float h, l, m;
  __device__ __forceinline__ void add(float f) {
    float t = __fadd_rn(h, f), b = __fsub_rn(t, h);
    const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(t, b)), __fsub_rn(f, b));
    h = t;
    t = __fadd_rn(l, e), b = __fsub_rn(t, l);
    m = __fadd_rn(m, __fadd_rn(__fsub_rn(l, __fsub_rn(t, b)), __fsub_rn(e, b)));
    l = t;
  }
};

// f_coarse_i(I, J) = w_i + mean over the cg x cg block of d_i(x - c_i).  A block
// of threads takes nc coarse nodes of a row: a thread sums one fine column (or
// every BF_T-th of them if cg > BF_T) of each direction over the cg rows, so
// that a warp reads 32 adjacent floats, and then one thread per direction and
// coarse node adds its columns.  Latency and issue of the sums bound it, next to
// the 36 B per fine node.  FP64 sums would need two operations per value at 1/64
// of the FP32 rate (by count about 60 us each at 2048^2), and one thread per
// coarse node left most of the chip idle.  A sum that is not finite in FP32 is
// taken again in FP64.
// Measured (GB300, us, cg = 8 / 4, one thread per coarse node before):
//   2048^2 183 / 175 -> 54 / 68      1000 x 1400  91 / 60 -> 23 / 27
//   32 x 256^2  83 / 93 -> 29 / 38   4096^2      599 / 611 -> 183 / 244
// (4096^2 is 91 us at the copy rate.)
constexpr int BF_T = 256;
constexpr int BF_MOST = BF_T + BF_T / 2;  // columns at stride cg | 1 (no bank conflicts)
__global__ void __launch_bounds__(BF_T)
    k_box_filter(const float *__restrict__ st, float *__restrict__ fc, int nx, int ny, int cg,
                 int nc, double inv) {
  __shared__ float part[3][Q][BF_MOST];
  const int NX = nx / cg, NY = ny / cg, tid = threadIdx.x;
  const int I0 = blockIdx.x * nc, J = blockIdx.y, b = blockIdx.z;
  const int n = min(nc, NX - I0), width = n * cg;
  const size_t plane = (size_t)nx * ny, cplane = (size_t)NX * NY;
  const float *base = st + (size_t)b * Q * plane;
  const int cols = min(cg, BF_T), stride = cols | 1;  // columns of a coarse node in `part`
  if (tid < width) {
    Sum3 s[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) s[i] = {0.f, 0.f, 0.f};
    for (int col = tid; col < width; col += BF_T) {
      const int x = I0 * cg + col;
      const int xs[3] = {wrap_index(x + 1, nx), x, wrap_index(x - 1, nx)};  // by c_x + 1
#pragma unroll 1  // two rows per body: 147 us instead of 55 (2048^2, cg = 8)
      for (int a = 0; a < cg; ++a) {
        const int y = J * cg + a;
        const size_t row[3] = {(size_t)wrap_index(y + 1, ny) * nx, (size_t)y * nx,
                               (size_t)wrap_index(y - 1, ny) * nx};
#pragma unroll
        for (int i = 0; i < Q; ++i)
          s[i].add(__ldg(base + i * plane + row[cy(i) + 1] + xs[cx(i) + 1]));
      }
    }
    const int at = tid / cols * stride + tid % cols;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      part[0][i][at] = s[i].h;
      part[1][i][at] = s[i].l;
      part[2][i][at] = s[i].m;
    }
  }
  __syncthreads();
  for (int o = tid; o < n * Q; o += BF_T) {
    const int i = o / n, k = o % n;
    Sum3 s = {0.f, 0.f, 0.f};
    for (int c = 0; c < cols; ++c) {
      s.add(part[0][i][k * stride + c]);
      s.add(part[1][i][k * stride + c]);
      s.m += part[2][i][k * stride + c];
    }
    double sum = (double)s.h + ((double)s.l + (double)s.m);
    if (!isfinite(s.h)) {
      sum = 0.0;
      for (int a = 0; a < cg; ++a) {
        const float *row =
            base + i * plane + (size_t)wrap_index(J * cg + a - cy(i), ny) * nx;
        for (int c = 0; c < cg; ++c)
          sum += (double)__ldg(row + wrap_index((I0 + k) * cg + c - cx(i), nx));
      }
    }
    fc[(size_t)b * Q * cplane + i * cplane + (size_t)J * NX + I0 + k] = (float)(sum * inv) + wf(i);
  }
}

// Velocity loss: per-node squared error, block partial sums (fixed order),
// and optionally dL/df_i = s ((u - u_t).(c_i - u)) / rho, s = 1/(N B).
__global__ void k_velocity_loss(const float *__restrict__ st, const float *__restrict__ utx,
                                const float *__restrict__ uty, float *__restrict__ partials,
                                float *__restrict__ dL_df, int nx, int ny, float s) {
  __shared__ float red[NT];
  int x, y, b;
  const bool ok = node_index(nx, x, y, b);
  float e = 0.0f;
  if (ok) {
    const size_t plane = (size_t)nx * ny;
    float d[Q];
    pull_node(st + (size_t)b * Q * plane, plane, nx, ny, x, y, d);
    const Moments m = node_moments(d);
    const size_t n = (size_t)b * plane + (size_t)y * nx + x;
    const float dx = m.ux - utx[n], dy = m.uy - uty[n];
    e = dx * dx + dy * dy;
    if (dL_df) {
      const float inv = s / m.rho;
      float *o = dL_df + (size_t)b * Q * plane + (size_t)y * nx + x;
#pragma unroll
      for (int i = 0; i < Q; ++i)
        o[i * plane] = inv * (dx * ((float)cx(i) - m.ux) + dy * ((float)cy(i) - m.uy));
    }
  }
  red[threadIdx.x] = e;
  __syncthreads();
  for (int w = NT / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    partials[((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = red[0];
}

// Single block: loss = scale * sum(partials), fixed order (strided then tree).
__global__ void k_sum_partials(const float *__restrict__ partials, int n, float scale,
                               float *loss) {
  __shared__ double red[256];
  double a = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) a += (double)partials[i];
  red[threadIdx.x] = a;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) loss[0] = (float)(red[0] * (double)scale);
}

// ---------------------------------------------------------------------------
// Losses on a node subset S (the training variant of SI section 2): one thread
// per listed node n = b*ny*nx + y*nx + x.  Per-sample errors in FP64, per-block
// FP64 partials (fixed order), then k_sum_partials_f64.  The gradient goes to
// the pre-collision field dL_df (zeroed beforehand by the launcher) with
// atomicAdd: distinct samples touch distinct entries, and a repeated sample
// adds the same value again, so the result does not depend on the order.
// An index outside [0, B ny nx) contributes nothing and sets bad_flag.
// ---------------------------------------------------------------------------
constexpr int SUB_THREADS = 256;

__device__ __forceinline__ bool decode_node(int n, int nx, int ny, int batch, int &x, int &y,
                                            int &b) {
  const long long plane = (long long)nx * ny;
  if (n < 0 || (long long)n >= plane * batch) return false;
  b = (int)(n / plane);
  const int r = (int)(n - (long long)b * plane);
  y = r / nx;
  x = r - y * nx;
  return true;
}

__device__ __forceinline__ void block_sum_f64(double e, double *__restrict__ partials) {
  __shared__ double red[SUB_THREADS];
  red[threadIdx.x] = e;
  __syncthreads();
  for (int w = SUB_THREADS / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) partials[blockIdx.x] = red[0];
}

// e = |u(n) - u_t(n)|^2 of the pre-collision populations at n;
// dL/df_i(n) = inv_count ((u - u_t).(c_i - u)) / rho   (L = sum e / (2 |S|)).
__global__ void __launch_bounds__(SUB_THREADS)
    k_velocity_loss_subset(const float *__restrict__ st, const int *__restrict__ idx, int count,
                           const float *__restrict__ utx, const float *__restrict__ uty,
                           double *__restrict__ partials, float *__restrict__ dL_df, int nx,
                           int ny, int batch, float inv_count, int *bad_flag) {
  const int s = blockIdx.x * SUB_THREADS + threadIdx.x;
  double e = 0.0;
  if (s < count) {
    int x, y, b;
    if (!decode_node(idx[s], nx, ny, batch, x, y, b)) {
      atomicOr(bad_flag, 1);
    } else {
      const size_t plane = (size_t)nx * ny;
      float d[Q];
      pull_node(st + (size_t)b * Q * plane, plane, nx, ny, x, y, d);
      const Moments m = node_moments(d);
      const size_t n = (size_t)b * plane + (size_t)y * nx + x;
      const float dx = m.ux - utx[n], dy = m.uy - uty[n];
      e = (double)dx * dx + (double)dy * dy;
      if (dL_df) {
        const float inv = inv_count / m.rho;
        float *o = dL_df + (size_t)b * Q * plane + (size_t)y * nx + x;
#pragma unroll
        for (int i = 0; i < Q; ++i)
          atomicAdd(o + i * plane, inv * (dx * ((float)cx(i) - m.ux) + dy * ((float)cy(i) - m.uy)));
      }
    }
  }
  block_sum_f64(e, partials);
}

// e = sum_i (g_i(n) - t_i(n))^2 with g the stored post-collision populations
// (g_i = state_i + w_i, formed in FP64) and t the target [b][i][y][x];
// dL/dg_i(n) = 2 (g_i - t_i) lands on the pre-collision entry it streams to,
// dL/df_i(n + c_i) (since f_i(x) = g_i(x - c_i)).
__global__ void __launch_bounds__(SUB_THREADS)
    k_population_loss_subset(const float *__restrict__ st, const int *__restrict__ idx, int count,
                             const float *__restrict__ target, double *__restrict__ partials,
                             float *__restrict__ dL_df, int nx, int ny, int batch,
                             int *bad_flag) {
  const int s = blockIdx.x * SUB_THREADS + threadIdx.x;
  double e = 0.0;
  if (s < count) {
    int x, y, b;
    if (!decode_node(idx[s], nx, ny, batch, x, y, b)) {
      atomicOr(bad_flag, 1);
    } else {
      const size_t plane = (size_t)nx * ny, base = (size_t)b * Q * plane;
      const size_t at = (size_t)y * nx + x;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const double d = ((double)st[base + i * plane + at] + (double)wf(i)) -
                         (double)target[base + i * plane + at];
        e += d * d;
        if (dL_df) {
          const int xs = wrap_index(x + cx(i), nx), ys = wrap_index(y + cy(i), ny);
          atomicAdd(dL_df + base + i * plane + (size_t)ys * nx + xs, (float)(2.0 * d));
        }
      }
    }
  }
  block_sum_f64(e, partials);
}

// Single block: loss = scale * sum(partials), fixed order (strided then tree).
__global__ void k_sum_partials_f64(const double *__restrict__ partials, int n, double scale,
                                   float *loss) {
  __shared__ double red[256];
  double a = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) a += partials[i];
  red[threadIdx.x] = a;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) loss[0] = (float)(red[0] * scale);
}

// Subsampling filter phi (SI section 2): the coarse node (I, J) takes the fine
// pre-collision populations at (cg I, cg J), f_i = state_i(x - c_i) + w_i.
__global__ void k_subsample(const float *__restrict__ st, float *__restrict__ fc, int nx, int ny,
                            int cg) {
  const int NX = nx / cg, NY = ny / cg;
  const int I = blockIdx.x * NT + threadIdx.x, J = blockIdx.y, b = blockIdx.z;
  if (I >= NX) return;
  const size_t plane = (size_t)nx * ny, cplane = (size_t)NX * NY;
  float d[Q];
  pull_node(st + (size_t)b * Q * plane, plane, nx, ny, I * cg, J * cg, d);
#pragma unroll
  for (int i = 0; i < Q; ++i)
    fc[(size_t)b * Q * cplane + i * cplane + (size_t)J * NX + I] = d[i] + wf(i);
}

// out_i(x) = in_i(x + DIR c_i), DIR = +1 push (transpose of the pull), -1 pull.
template <int DIR>
__global__ void k_shift(const float *__restrict__ in, float *__restrict__ out, int nx, int ny) {
  int x, y, b;
  if (!node_index(nx, x, y, b)) return;
  const size_t plane = (size_t)nx * ny, base = (size_t)b * Q * plane;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int xs = wrap_index(x + DIR * cx(i), nx), ys = wrap_index(y + DIR * cy(i), ny);
    out[base + i * plane + (size_t)y * nx + x] = in[base + i * plane + (size_t)ys * nx + xs];
  }
}

}  // namespace

// Steps per launch: whichever of the three forms has the least estimated time per
// step, from the sizes alone.  The estimates are fits to measurements (GB300, us
// per step; 60 shapes of 4 k to 4 M nodes, within about 25 % of them):
//   single steps  2.4 (4-node threads; 1.5 one-node) plus 8 ps per node in L2, 10
//                 one-node, 11.6 from HBM, and at least 2.4 (1.1) ns per block, of 512
//                 (128) nodes of one row: narrow lattices have many blocks;
//   k_steps_tile  t = 3: 1.0 + 0.54 per wave of one region per SM, 5.2 ns per region
//                 beyond three; a region stores 60 x 12 nodes, and computes 64 x 16
//                 however few of them the lattice has;
//   k_steps_small t = 8: 0.6 + 1.9 ns per 8 x 8 tile, up to 128^2 nodes.
// So squares and batches of small lattices take several steps per launch (64^2: 2.9
// -> 0.7 us per step, 256 lattices of 64^2: 40 -> 15, 64 x 16384: 40 -> 13), and
// lattices a row or two high do not: 65536 x 2 takes 3.5 us by single steps and 6.1 by
// the tile kernel, 16384 x 1 takes 3.0, 2.6 and (small kernel) 4.2.  The tile kernel has
// to be 5 % better: with equal estimates (61 x 1000) its Smagorinsky form is slower.
// Plane offsets of all forms are 32-bit (lbm_init refuses planes of 2^31 nodes).
StepPlan step_plan(const Grid &g) {
  const double nodes = (double)g.nodes(), rows = (double)g.ny * g.batch;
  auto over = [](int n, int d) { return (double)((n + d - 1) / d); };
  const bool vec = g.nx % 4 == 0;
  const double per_node = nodes > 1.5e6 ? 11.6e-6 : (vec ? 8e-6 : 10e-6);
  const double single = std::max((vec ? 2.4 : 1.5) + per_node * nodes,
                                 vec ? 2.4e-3 * over(g.nx, 4 * VEC_THREADS) * rows
                                     : 1.1e-3 * over(g.nx, SCALAR_THREADS) * rows);
  constexpr int RING = 2 * (MT_MOST - 1), TS = 8;
  const double regions = over(g.nx, MT_X - RING) * over(g.ny, MT_Y - RING) * g.batch;
  const double waves = std::ceil(regions / 152);
  const double tile = std::max(1.0 + 0.54 * std::min(waves, 3.0), 5.2e-3 * regions);
  const double small = 0.6 + 1.9e-3 * over(g.nx, TS) * over(g.ny, TS) * g.batch;
  if (nodes <= 128 * 128 && small <= single && small <= tile) return {8, TS};
  if (1.05 * tile <= single) return {MT_MOST, 0};
  return {1, 0};
}

cudaError_t launch_steps_bgk(const Grid &g, const float *in, float *out, const CollideParams &p,
                             int t, int *flag, cudaStream_t s) {
  return launch_steps<KIND_BGK>(g, in, out, p, t, flag, s);
}

cudaError_t launch_steps_smag(const Grid &g, const float *in, float *out, const CollideParams &p,
                              int t, int *flag, cudaStream_t s) {
  return launch_steps<KIND_SMAG>(g, in, out, p, t, flag, s);
}

cudaError_t launch_set_state(const Grid &g, const float *f_pre, float *state, cudaStream_t s) {
  k_set_state<<<node_grid(g), NT, 0, s>>>(f_pre, state, g.nx, g.ny);
  return cudaGetLastError();
}

cudaError_t launch_get_state(const Grid &g, const float *state, float *f_pre, cudaStream_t s) {
  k_get_state<<<node_grid(g), NT, 0, s>>>(state, f_pre, g.nx, g.ny);
  return cudaGetLastError();
}

cudaError_t launch_init_equilibrium(const Grid &g, const float *rho, const float *ux,
                                    const float *uy, float *state, cudaStream_t s) {
  k_init_equilibrium<<<node_grid(g), NT, 0, s>>>(rho, ux, uy, state, g.nx, g.ny);
  return cudaGetLastError();
}

cudaError_t launch_moments(const Grid &g, const float *state, float *rho, float *ux, float *uy,
                           cudaStream_t s) {
  k_moments<<<node_grid(g), NT, 0, s>>>(state, rho, ux, uy, g.nx, g.ny);
  return cudaGetLastError();
}

cudaError_t launch_box_filter(const Grid &g, const float *state, int cg, float *f_coarse,
                              cudaStream_t s) {
  // a block of one node is that node: the same values in half the time (1024^2: 126 us
  // as sums; 88 with one thread per coarse node)
  if (cg == 1) return launch_subsample(g, state, cg, f_coarse, s);
  const int nc = cg < BF_T ? BF_T / cg : 1, NX = g.nx / cg;
  dim3 grid((NX + nc - 1) / nc, g.ny / cg, g.batch);
  k_box_filter<<<grid, BF_T, 0, s>>>(state, f_coarse, g.nx, g.ny, cg, nc,
                                     1.0 / ((double)cg * cg));
  return cudaGetLastError();
}

int loss_partials(const Grid &g) { return (int)(((g.nx + NT - 1) / NT) * (size_t)g.ny * g.batch); }

cudaError_t launch_velocity_loss(const Grid &g, const float *state, const float *utx,
                                 const float *uty, float *partials, float *loss, float *dL_df,
                                 cudaStream_t s) {
  const float inv_nb = (float)(1.0 / ((double)g.plane() * g.batch));
  k_velocity_loss<<<node_grid(g), NT, 0, s>>>(state, utx, uty, partials, dL_df, g.nx, g.ny,
                                              inv_nb);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_sum_partials<<<1, 256, 0, s>>>(partials, loss_partials(g), 0.5f * inv_nb, loss);
  return cudaGetLastError();
}

int subset_partials(int count) { return (count + SUB_THREADS - 1) / SUB_THREADS; }

cudaError_t launch_velocity_loss_subset(const Grid &g, const float *state, const int *idx,
                                        int count, const float *utx, const float *uty,
                                        double *partials, float *loss, float *dL_df,
                                        int *bad_flag, cudaStream_t s) {
  if (dL_df) {
    cudaError_t e = cudaMemsetAsync(dL_df, 0, g.state_floats() * sizeof(float), s);
    if (e != cudaSuccess) return e;
  }
  const int blocks = subset_partials(count);
  k_velocity_loss_subset<<<blocks, SUB_THREADS, 0, s>>>(state, idx, count, utx, uty, partials,
                                                        dL_df, g.nx, g.ny, g.batch,
                                                        (float)(1.0 / count), bad_flag);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_sum_partials_f64<<<1, 256, 0, s>>>(partials, blocks, 0.5 / count, loss);
  return cudaGetLastError();
}

cudaError_t launch_population_loss_subset(const Grid &g, const float *state, const int *idx,
                                          int count, const float *target, double *partials,
                                          float *loss, float *dL_df, int *bad_flag,
                                          cudaStream_t s) {
  if (dL_df) {
    cudaError_t e = cudaMemsetAsync(dL_df, 0, g.state_floats() * sizeof(float), s);
    if (e != cudaSuccess) return e;
  }
  const int blocks = subset_partials(count);
  k_population_loss_subset<<<blocks, SUB_THREADS, 0, s>>>(state, idx, count, target, partials,
                                                          dL_df, g.nx, g.ny, g.batch, bad_flag);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_sum_partials_f64<<<1, 256, 0, s>>>(partials, blocks, 1.0, loss);
  return cudaGetLastError();
}

cudaError_t launch_subsample(const Grid &g, const float *state, int cg, float *f_coarse,
                             cudaStream_t s) {
  dim3 grid((g.nx / cg + NT - 1) / NT, g.ny / cg, g.batch);
  k_subsample<<<grid, NT, 0, s>>>(state, f_coarse, g.nx, g.ny, cg);
  return cudaGetLastError();
}

cudaError_t launch_push(const Grid &g, const float *in, float *out, cudaStream_t s) {
  k_shift<1><<<node_grid(g), NT, 0, s>>>(in, out, g.nx, g.ny);
  return cudaGetLastError();
}

cudaError_t launch_pull(const Grid &g, const float *in, float *out, cudaStream_t s) {
  k_shift<-1><<<node_grid(g), NT, 0, s>>>(in, out, g.nx, g.ny);
  return cudaGetLastError();
}

}  // namespace lbm
