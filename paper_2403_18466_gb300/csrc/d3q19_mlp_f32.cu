// d3q19_mlp_f32.cu -- the paper's learned collision on D3Q19 in FP32 on the
// CUDA cores (19 -> 300 -> 300 -> 100 -> 19, LeakyReLU, conservation layer),
// fused with the pull-stream, the BGK update and the EDM forcing: the
// reference path of the tensor-core kernel.
//
// What bounds it: 127.6 k FMA per node, so the FP32 pipe.  Each layer is a
// register-tiled matrix product over a tile of 32 consecutive nodes of the
// flattened lattice (so no lane is lost at the ends of rows): a thread holds
// 8 nodes x 10 units, each with the sums over the even and the odd inputs in
// one packed f32x2 accumulator, and per pair of inputs reads 8 activation
// pairs and 10 weight pairs with 9 16-byte shared-memory loads for 80 packed
// FMAs.  (The packed form does not raise the pipe's rate, it halves the issue
// slots; pairing the inputs needs no duplicated operands.)  The two long
// layers add the sums of their two halves at the end, so every output is the
// sum of four chains of 75 (25) inputs and the bias.  The activations of a
// layer live in shared memory as [k / 2][node][2] and are replaced in place
// once every thread has its sums in registers; the weights, laid out as
// [k / 2][unit][2] by k3_prepare_weights_f32, stream through a two-stage
// cp.async buffer in chunks of KC inputs.
// Measured (GB300, 32^3, one step): 224 us = 37 TFLOP/s, FMA pipe 58 % and
// shared-memory pipe 51 % busy, two warps per scheduler (246 registers); one
// output per lane with a scalar weight load per FMA took 2,640 us.  Units
// instead of inputs paired (8 x 20 units per thread, one chain per output)
// ran at 200 us with 2.6 times the rounding error of this form in o.
#include <cstdint>

#include "d3q19.cuh"
#include "kernels3d.h"

namespace lbm {
namespace d3 {
namespace {

constexpr int THREADS = 128;
constexpr int M = 32;           // nodes per tile
constexpr int KC = 10;          // inputs per staged chunk
constexpr int NU = 320;         // padded units of layers 1 and 2 (5 groups of 64)
constexpr int NU3 = 128;        // padded units of layer 3
constexpr int NU4 = 20;         // padded outputs
constexpr int K1 = 20;          // padded inputs of layer 1
static_assert(H1 % (2 * KC) == 0 && H2 % (2 * KC) == 0 && K1 % KC == 0 && KC % 2 == 0 &&
                  H3 % 4 == 0,
              "chunking");

// Prepared weights (floats): every layer as [k / 2][unit][k % 2], zero padded.
constexpr int P_W1 = 0;
constexpr int P_W2 = P_W1 + K1 * NU;
constexpr int P_W3 = P_W2 + H1 * NU;
constexpr int P_W4 = P_W3 + H2 * NU3;
constexpr int P_B1 = P_W4 + H3 * NU4;
constexpr int P_B2 = P_B1 + NU;
constexpr int P_B3 = P_B2 + NU;
constexpr int P_B4 = P_B3 + NU3;
constexpr int P_TOTAL = P_B4 + NU4;

__global__ void k3_prepare_weights_f32(Mlp3 w, float *__restrict__ p) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < P_TOTAL; e += gridDim.x * blockDim.x) {
    float v = 0.f;
    if (e < P_W2) {
      const int f = e - P_W1, k = f / (2 * NU) * 2 + f % 2, n = f / 2 % NU;
      if (k < Q && n < H1) v = w.w1[n * Q + k];
    } else if (e < P_W3) {
      const int f = e - P_W2, k = f / (2 * NU) * 2 + f % 2, n = f / 2 % NU;
      if (n < H2) v = w.w2[n * H1 + k];
    } else if (e < P_W4) {
      const int f = e - P_W3, k = f / (2 * NU3) * 2 + f % 2, n = f / 2 % NU3;
      if (n < H3) v = w.w3[n * H2 + k];
    } else if (e < P_B1) {
      const int f = e - P_W4, k = f / (2 * NU4) * 2 + f % 2, n = f / 2 % NU4;
      if (n < Q) v = w.w4[n * H3 + k];
    } else if (e < P_B2) {
      if (e - P_B1 < H1) v = w.b1[e - P_B1];
    } else if (e < P_B3) {
      if (e - P_B2 < H2) v = w.b2[e - P_B2];
    } else if (e < P_B4) {
      if (e - P_B3 < H3) v = w.b3[e - P_B3];
    } else {
      if (e - P_B4 < Q) v = w.b4[e - P_B4];
    }
    p[e] = v;
  }
}

// The staged chunks in the order they are used: layer 1 (2), layer 2 (30),
// layer 3 (30), layer 4 (1).
constexpr int C_L2 = K1 / KC, C_L3 = C_L2 + H1 / KC, C_L4 = C_L3 + H2 / KC, CHUNKS = C_L4 + 1;
constexpr int STAGE = KC * NU;  // floats of one stage
static_assert(H3 * NU4 <= STAGE && KC * NU3 <= STAGE, "stage size");

struct Smem {
  float h[H1 / 2][2 * M];            // activations [k / 2][node][k % 2]
  float stage[2][STAGE];             // weight chunks
  float4 half[NU / 16][THREADS];     // each thread's sums of the first half of the inputs
};

__device__ __forceinline__ void stage_chunk(const float *__restrict__ p, int c, float *dst) {
  int off, n;  // floats
  if (c < C_L3) {
    off = c * STAGE, n = STAGE;  // W1 and W2 are contiguous
  } else if (c < C_L4) {
    off = P_W3 + (c - C_L3) * (KC * NU3), n = KC * NU3;
  } else {
    off = P_W4, n = H3 * NU4;
  }
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  for (int e = threadIdx.x; e < n / 4; e += THREADS)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16 * e), "l"(p + off + 4 * e)
                 : "memory");
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// Chunk c has landed and every thread is done with chunk c - 1, whose stage
// the next chunk may take.
__device__ __forceinline__ void next_chunk(const float *__restrict__ p, int c, float (*stage)[STAGE]) {
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  if (c + 1 < CHUNKS) stage_chunk(p, c + 1, stage[(c + 1) & 1]);
}

// One hidden layer of 64 NG padded units: CHUNKS_L staged chunks from number c
// on, in place on s.h.  Thread (ng, ug) owns nodes 8 j + 2 ng, + 1 (j < 4) and
// units 64 q + 2 ug, + 1 (q < NG).
template <int NG, int CHUNKS_L>
__device__ __forceinline__ void hidden_layer(Smem &s, const float *__restrict__ p, int c,
                                             const float *__restrict__ bias, int units, int ng,
                                             int ug) {
  constexpr bool HALVES = CHUNKS_L % 2 == 0 && CHUNKS_L > 2;
  float2 acc[NG][2][8];
#pragma unroll
  for (int q = 0; q < NG; ++q)
#pragma unroll
    for (int n = 0; n < 8; ++n) acc[q][0][n] = acc[q][1][n] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int e = 0; e < CHUNKS_L; ++e, ++c) {
    if (HALVES && e == CHUNKS_L / 2) {
#pragma unroll
      for (int q = 0; q < NG; ++q)
#pragma unroll
        for (int n = 0; n < 8; n += 2) {
          s.half[4 * q + n / 2][threadIdx.x] =
              make_float4(acc[q][0][n].x + acc[q][0][n].y, acc[q][1][n].x + acc[q][1][n].y,
                          acc[q][0][n + 1].x + acc[q][0][n + 1].y,
                          acc[q][1][n + 1].x + acc[q][1][n + 1].y);
          acc[q][0][n] = acc[q][1][n] = make_float2(0.f, 0.f);
          acc[q][0][n + 1] = acc[q][1][n + 1] = make_float2(0.f, 0.f);
        }
    }
    next_chunk(p, c, s.stage);
    const float *w = s.stage[c & 1] + 4 * ug;
    const float *h = &s.h[e * (KC / 2)][4 * ng];
#pragma unroll
    for (int k = 0; k < KC / 2; ++k) {
      float2 a[8];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 v = *reinterpret_cast<const float4 *>(h + k * 2 * M + 16 * j);
        a[2 * j] = make_float2(v.x, v.y);
        a[2 * j + 1] = make_float2(v.z, v.w);
      }
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        const float4 v = *reinterpret_cast<const float4 *>(w + k * (128 * NG) + 128 * q);
        const float2 w0 = make_float2(v.x, v.y), w1 = make_float2(v.z, v.w);
#pragma unroll
        for (int n = 0; n < 8; ++n) {
          acc[q][0][n] = __ffma2_rn(w0, a[n], acc[q][0][n]);
          acc[q][1][n] = __ffma2_rn(w1, a[n], acc[q][1][n]);
        }
      }
    }
  }
  __syncthreads();  // every thread has read the layer's input
#pragma unroll
  for (int q = 0; q < NG; ++q) {
    const int row = 32 * q + ug;
    if (2 * row >= units) continue;
    const float2 b = __ldg(reinterpret_cast<const float2 *>(bias) + row);
#pragma unroll
    for (int n = 0; n < 8; n += 2) {
      float v[4] = {acc[q][0][n].x + acc[q][0][n].y, acc[q][1][n].x + acc[q][1][n].y,
                    acc[q][0][n + 1].x + acc[q][0][n + 1].y,
                    acc[q][1][n + 1].x + acc[q][1][n + 1].y};
      if (HALVES) {
        const float4 t = s.half[4 * q + n / 2][threadIdx.x];
        v[0] += t.x, v[1] += t.y, v[2] += t.z, v[3] += t.w;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float a = (j & 1 ? b.y : b.x) + v[j];
        v[j] = a >= 0.f ? a : LEAKY * a;
      }
      *reinterpret_cast<float4 *>(&s.h[row][8 * n + 4 * ng]) = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
}

struct Node {
  long long n;  // flattened index within the lattice
  int x, y, z, b;
};
__device__ __forceinline__ Node locate(const Grid3 &g, long long n) {
  const long long vol = (long long)g.nx * g.ny * g.nz;
  Node p;
  p.b = (int)(n / vol);
  p.n = n - p.b * vol;
  const long long row = p.n / g.nx;
  p.x = (int)(p.n - row * g.nx);
  p.z = (int)(row / g.ny);
  p.y = (int)(row - (long long)p.z * g.ny);
  return p;
}
__device__ __forceinline__ void pull(const float *__restrict__ in, const Grid3 &g, const Node &p,
                                     float d[Q]) {
  const size_t vol = g.volume();
  const float *gb = in + (size_t)p.b * Q * vol;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    int xs = p.x - cx(i), ys = p.y - cy(i), zs = p.z - cz(i);
    xs = xs < 0 ? xs + g.nx : (xs >= g.nx ? xs - g.nx : xs);
    ys = ys < 0 ? ys + g.ny : (ys >= g.ny ? ys - g.ny : ys);
    zs = zs < 0 ? zs + g.nz : (zs >= g.nz ? zs - g.nz : zs);
    d[i] = __ldg(gb + (size_t)i * vol + ((size_t)zs * g.ny + ys) * g.nx + xs);
  }
}

__global__ void __launch_bounds__(THREADS, 2)
    k3_step_mlp_f32(const float *__restrict__ in, float *__restrict__ out, Grid3 g, Collide3 c,
                    const float *__restrict__ p, long long nodes, int *flag) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem &s = *reinterpret_cast<Smem *>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ng = lane & 3, ug = 8 * warp + (lane >> 2);
  stage_chunk(p, 0, s.stage[0]);
  const long long node = (long long)blockIdx.x * M + lane;
  const bool live = warp == 0 && node < nodes;
  if (warp == 0) {
    float d[Q], deq[Q];
    float inv = 1.f;
    if (live) {
      pull(in, g, locate(g, node), d);
      const Moments m = node_moments(d);
      shifted_feq(m, deq);
      inv = 1.0f / m.rho;
    }
#pragma unroll
    for (int i = 0; i < K1; ++i)
      s.h[i / 2][2 * lane + i % 2] = i < Q && live ? (d[i] - deq[i]) * inv : 0.f;
  }
  hidden_layer<NU / 64, C_L2>(s, p, 0, p + P_B1, H1, ng, ug);
  hidden_layer<NU / 64, C_L3 - C_L2>(s, p, C_L2, p + P_B2, H2, ng, ug);
  hidden_layer<NU3 / 64, C_L4 - C_L3>(s, p, C_L3, p + P_B3, H3, ng, ug);
  next_chunk(p, C_L4, s.stage);
  {
    // output layer (1.5 % of the FMAs): one node and 5 outputs per thread, the
    // inputs in four chains
    const float *w = s.stage[C_L4 & 1] + 10 * warp;
    float2 acc[2][5];
#pragma unroll
    for (int i = 0; i < 5; ++i) acc[0][i] = acc[1][i] = make_float2(0.f, 0.f);
    for (int k = 0; k < H3 / 2; k += 2)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float2 h = *reinterpret_cast<const float2 *>(&s.h[k + j][2 * lane]);
#pragma unroll
        for (int i = 0; i < 5; ++i)
          acc[j][i] = __ffma2_rn(
              *reinterpret_cast<const float2 *>(w + (k + j) * 2 * NU4 + 2 * i), h, acc[j][i]);
      }
    // rows from H3 / 2 on are no longer read
#pragma unroll
    for (int i = 0; i < 5; ++i)
      s.h[H3 / 2 + 5 * warp + i][lane] = __ldg(p + P_B4 + 5 * warp + i) +
                                         ((acc[0][i].x + acc[0][i].y) + (acc[1][i].x + acc[1][i].y));
  }
  __syncthreads();
  if (!live) return;
  const Node at = locate(g, node);
  float d[Q], deq[Q], o[Q];
  pull(in, g, at, d);
  const Moments m = node_moments(d);
  shifted_feq(m, deq);
#pragma unroll
  for (int i = 0; i < Q; ++i) o[i] = s.h[H3 / 2 + i][lane];
  project(o);
  const float scale = m.rho * c.omega;
#pragma unroll
  for (int i = 0; i < Q; ++i) d[i] += c.omega * (deq[i] - d[i]) + scale * o[i];
  add_edm_force(m, c.fx_y ? c.fx_y[at.y] : 0.f, c.fy_z ? c.fy_z[at.z] : 0.f,
                c.fz_x ? c.fz_x[at.x] : 0.f, d);
  const unsigned mask = __ballot_sync(__activemask(), is_unstable(m));
  if (mask && lane == __ffs(mask) - 1 && *reinterpret_cast<volatile int *>(flag) == 0)
    atomicOr(flag, 1);
  const size_t vol = g.volume();
  float *op = out + (size_t)at.b * Q * vol + at.n;
#pragma unroll
  for (int i = 0; i < Q; ++i) op[(size_t)i * vol] = d[i];
}

}  // namespace

size_t mlp_f32_weight_floats() { return P_TOTAL; }

cudaError_t launch_prepare_weights_f32(const Mlp3 &w, float *p, cudaStream_t s) {
  k3_prepare_weights_f32<<<(P_TOTAL + 255) / 256, 256, 0, s>>>(w, p);
  return cudaGetLastError();
}

cudaError_t launch_step_mlp_f32(const Grid3 &g, const float *in, float *out, const Collide3 &c,
                                const float *p, int *flag, cudaStream_t s) {
  const cudaError_t e = cudaFuncSetAttribute(
      k3_step_mlp_f32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
  if (e != cudaSuccess) return e;
  const long long nodes = (long long)g.nodes(), tiles = (nodes + M - 1) / M;
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  k3_step_mlp_f32<<<(unsigned)tiles, THREADS, sizeof(Smem), s>>>(in, out, g, c, p, nodes, flag);
  return cudaGetLastError();
}

}  // namespace d3
}  // namespace lbm
