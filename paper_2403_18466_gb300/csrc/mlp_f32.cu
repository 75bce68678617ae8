// mlp_f32.cu -- fused pull-stream + learned collision, all in FP32 on the
// CUDA cores (the correctness companion of the tensor-core kernel).
//
// Per node (Eq. S10-S12 with the network of this library):
//   x     = (f - feq) / rho                     (9, intensive input)
//   h1    = tanh(W1 x + b1), h2 = tanh(W2 h1 + b2), o = W3 h2 + b3
//   ohat  = o - mean(o) - c_x (sum o c_x)/6 - c_y (sum o c_y)/6   (Eqs. S11-S12, D2Q9)
//   f'    = f + (feq - f)/tau + (rho/tau) ohat + f_ext            (Eq. S10, Eq. S5)
// About 5.3 k FMAs and 128 tanh per node bound it to the FP32 pipe.  A block of
// 128 threads owns tiles of 128 consecutive nodes of the flattened lattice (no
// lane is lost at the ends of rows): per node one thread forms x and the BGK +
// force update, the layers are matrix products over the tile (8 nodes x 8 units
// per thread, dense_f32.cuh), and the activations stay in shared memory, each
// layer's in place of its input's.
// Measured (GB300): 3.00 G nodes/s at 2048^2, 2.73 at 4 x 333 x 250, 33 us per
// step at 256^2 and 16 at 64^2, against 3.01, 2.03, 96 and 90 with one node per
// thread and tanhf; FMA pipe ~60 % busy.  The error of the learned correction
// against 64 bits fell from 1.9e-7 to 1.2 - 1.5e-7.  (tanh2's accuracy and what
// it costs stand beside it.)
#include "dense_f32.cuh"
#include "kernels.h"

namespace lbm {
namespace {

using namespace f32;

constexpr int BLOCKS_PER_SM = 2;  // of 205 registers per thread; three spill and are 24 % slower

struct __align__(16) Smem {
  float w1[HIDDEN][XS];  // [j][k], b1 at k = 9, zeros
  float w2[HIDDEN][HS];
  float w3[XS][HS];      // rows 9..11 zero
  float b2[HIDDEN];
  float b3[XS];
  float x[TILE][XS];     // x | 1 | 0 0, later the outputs
  float h[TILE][HS];     // h1, then h2
  float base[Q + 1][TILE];  // BGK + force update of the tile's nodes, rho/tau
};

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

__global__ void __launch_bounds__(TILE, BLOCKS_PER_SM)
    k_step_mlp_f32(const float *__restrict__ in, float *__restrict__ out, int nx, int ny,
                   long long nodes, CollideParams p, MlpF32 w, int *flag) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem &S = *reinterpret_cast<Smem *>(smem_raw);
  const int t = threadIdx.x;
  for (int e = t; e < HIDDEN * XS; e += TILE) {
    const int j = e / XS, k = e % XS;
    S.w1[j][k] = k < 9 ? w.w1[j * 9 + k] : (k == 9 ? w.b1[j] : 0.f);
  }
  for (int e = t; e < HIDDEN * HIDDEN; e += TILE) S.w2[e / HIDDEN][e % HIDDEN] = w.w2[e];
  for (int e = t; e < XS * HIDDEN; e += TILE)
    S.w3[e / HIDDEN][e % HIDDEN] = e < 9 * HIDDEN ? w.w3[e] : 0.f;
  if (t < HIDDEN) S.b2[t] = w.b2[t];
  if (t < XS) S.b3[t] = t < 9 ? w.b3[t] : 0.f;
  // GEMM layout: units i * 8 + ug and nodes i * 16 + ng (hidden layers), outputs
  // i * 4 + og and nodes i * 32 + ngo (last layer)
  const int ug = t & 7, ng = t >> 3, og = t & 3, ngo = t >> 2;
  const size_t plane = (size_t)nx * ny;
  bool bad = false;
  for (long long tile = blockIdx.x; tile * TILE < nodes; tile += gridDim.x) {
    const long long n = tile * TILE + t;
    const bool active = n < nodes;
    size_t at = 0;  // of population 0 of this node
    if (active) {
      const int b = (int)(n / (long long)plane);
      const long long r = n - b * (long long)plane;
      const int y = (int)(r / nx), x = (int)(r - (long long)y * nx);
      at = (size_t)b * Q * plane + (size_t)r;
      const float *gb = in + (size_t)b * Q * plane;
      const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
      const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
      float d[Q], deq[Q], xin[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const int xs = cx(i) == 0 ? x : (cx(i) == 1 ? xm : xp);
        const int ys = cy(i) == 0 ? y : (cy(i) == 1 ? ym : yp);
        d[i] = __ldg(gb + i * plane + (size_t)ys * nx + xs);
      }
      const Moments m = node_moments(d);
      bad |= is_unstable(m);
      shifted_feq(m, deq);
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        xin[i] = (d[i] - deq[i]) * m.inv_rho;
        d[i] = bgk_relax(d[i], deq[i], p.omega);
      }
      add_edm_force_x(m, p.force ? __ldg(p.force + y) : 0.0f, d);
#pragma unroll
      for (int i = 0; i < Q; ++i) S.base[i][t] = d[i];
      S.base[Q][t] = m.rho * p.omega;
      float4 *xr = reinterpret_cast<float4 *>(&S.x[t][0]);
      xr[0] = make_float4(xin[0], xin[1], xin[2], xin[3]);
      xr[1] = make_float4(xin[4], xin[5], xin[6], xin[7]);
      xr[2] = make_float4(xin[8], 1.0f, 0.f, 0.f);
    } else {
#pragma unroll
      for (int k = 0; k < XS; ++k) S.x[t][k] = 0.f;
    }
    __syncthreads();
    // h1 = tanh(W1 x + b1), then h2 = tanh(W2 h1 + b2) in its place (one copy of
    // the epilogue for both, for the instruction cache)
#pragma unroll 1
    for (int layer = 1; layer <= 2; ++layer) {
      float2 acc[8][8];
      clear(acc);
      if (layer == 1)
        dense_acc<8, 8, XS / 4, XS, XS>(&S.x[ng][0], 16, &S.w1[ug][0], 8, acc);
      else
        dense_acc<8, 8, HIDDEN / 4, HS, HS>(&S.h[ng][0], 16, &S.w2[ug][0], 8, acc);
      if (layer == 2) __syncthreads();  // h1 is read
#pragma unroll
      for (int c = 0; c < 8; c += 2) {
        const float2 bias = layer == 1 ? make_float2(0.f, 0.f)
                                       : make_float2(S.b2[c * 8 + ug], S.b2[c * 8 + 8 + ug]);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const float2 h =
              tanh2(__fadd2_rn(make_float2(total(acc[r][c]), total(acc[r][c + 1])), bias));
          S.h[r * 16 + ng][c * 8 + ug] = h.x;
          S.h[r * 16 + ng][c * 8 + 8 + ug] = h.y;
        }
      }
      __syncthreads();
    }
    {
      float2 acc[4][3];
      clear(acc);
      dense_acc<4, 3, HIDDEN / 4, HS, HS>(&S.h[ngo][0], 32, &S.w3[og][0], 4, acc);
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) S.x[r * 32 + ngo][c * 4 + og] = total(acc[r][c]) + S.b3[c * 4 + og];
    }
    __syncthreads();
    if (active) {
      float o[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) o[i] = S.x[t][i];
      project9(o);
      const float rw = S.base[Q][t];  // rho / tau
#pragma unroll
      for (int i = 0; i < Q; ++i) out[at + i * plane] = fmaf(rw, o[i], S.base[i][t]);
    }
  }
  flag_unstable(bad, flag);
}

}  // namespace

cudaError_t launch_step_mlp_f32(const Grid &g, const float *in, float *out,
                                const CollideParams &p, const MlpF32 &w, int sms, int *flag,
                                cudaStream_t s) {
  const cudaError_t e = allow_smem(k_step_mlp_f32, sizeof(Smem));
  if (e != cudaSuccess) return e;
  const long long slots = (long long)BLOCKS_PER_SM * sms;
  const long long nodes = (long long)g.nodes(), tiles = (nodes + TILE - 1) / TILE;
  k_step_mlp_f32<<<(unsigned)(tiles < slots ? tiles : slots), TILE, sizeof(Smem), s>>>(
      in, out, g.nx, g.ny, nodes, p, w, flag);
  return cudaGetLastError();
}

}  // namespace lbm
