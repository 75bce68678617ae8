// adjoint.cu -- hand-written reverse mode of one unrolled step of the
// learned-collision lattice Boltzmann model (unrolled training, SI section 2),
// FP32 on the CUDA cores, and the deterministic weight-gradient reduction.
//
// Forward step (the one being differentiated): g'(x) = C(f(x)) with the
// pull f_i(x) = g_i(x - c_i) and C the learned collision of Eq. S10-S12 plus
// the EDM force (Eq. S5).  Given lam' = dL/dg', the adjoint step computes
//   lam_i(x - c_i) = [J_C(f(x))^T lam'(x)]_i        (transpose of the pull = push)
//   dtheta        += sum_x (dC/dtheta)^T lam'(x)
//
// About 16 k FMAs per node bound it to the FP32 pipe: the forward layers, the
// products with the transposed weights, and the weight-gradient sums, all as
// matrix products over tiles of 128 consecutive nodes of the flattened lattice
// in packed f32x2 arithmetic (dense_f32.cuh).  A CTA (one per SM) has two
// groups of 128 threads with a tile and its buffers each, so that one group's
// node work and barriers run beside the other's products; the weights are
// shared.  Per tile:
//   x, dL/do = P (rho omega lam')        one node per thread
//   h1, h2 = tanh(...)                   8 nodes x 8 units per thread
//   dW3 += dL/do^T h2
//   dL/da2 = (dL/do W3)(1 - h2^2)        in place of h2
//   dW2 += dL/da2^T h1                   8 x 4 entries per thread
//   dL/da1 = (dL/da2 W2)(1 - h1^2)       in place of dL/da2
//   dW1 += dL/da1^T [x | 1], dL/dx = dL/da1 W1
//   the rest of the chain rule and the scatter of lam, one node per thread
// The output o is not recomputed: the update needs it only in the
// rho-derivative of its scaling, sum_i lam'_i omega (P o)_i = (dL/do . o)/rho, and
// dL/do . o = (dL/do W3) . h2 + dL/do . b3, which the third product yields.
// Sums over nodes run tile by tile and then over a group's tiles; each CTA
// writes its own row of partial sums, and a second kernel adds the rows in a
// fixed order, so dtheta is bitwise reproducible.
// Measured (GB300): a training step of 8 x 256^2 trajectories, 16 steps, from
// 17.3 to 11.9 ms with the forward of mlp_f32.cu (one node per thread, 128
// threads per SM, before).
#include "adjoint_node.cuh"
#include "dense_f32.cuh"
#include "kernels.h"
#include "umma.cuh"

namespace lbm {
namespace {

using namespace f32;

constexpr int GROUPS = 2;
constexpr int THREADS = GROUPS * TILE;
constexpr int SMALL = 20;  // running sums per thread: dW1 | db1 (10), dW3 (9), db2

struct __align__(16) Group {
  float h1[TILE][HS];
  float h2[TILE][HS];  // h2, then dL/da2, then dL/da1
  float x[TILE][XS];   // x | 1 | 0 0
  float ob[TILE][XS];  // dL/do | 0, then dL/dx
  float small[SMALL][TILE];
  float dot[TILE];     // (dL/do W3) . h2
};
struct __align__(16) AdjSmem {
  float w1[HIDDEN][XS];   // [j][k], b1 at k = 9, zeros
  float w1t[XS][HS];      // [k][j], rows 9..11 zero
  float w2[HIDDEN][HS];   // [j][k]
  float w2t[HIDDEN][HS];  // [k][j]
  float w3t[HIDDEN][XS];  // [j][i], zeros
  float b2[HIDDEN];
  float b3[XS];
  Group g[GROUPS];
};
static_assert(sizeof(AdjSmem) <= 227 * 1024, "shared memory layout too large");
static_assert(sizeof(float) * NPARAMS <= sizeof(float) * TILE * HS, "a group's sums fit its h1");

__global__ void __launch_bounds__(THREADS, 1)
    k_adjoint_step(const float *__restrict__ state, const float *__restrict__ lam_next,
                   float *__restrict__ lam_out, int nx, int ny, long long nodes, CollideParams p,
                   MlpF32 w, float *__restrict__ partials, int accumulate) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  AdjSmem &S = *reinterpret_cast<AdjSmem *>(smem_raw);
  for (int e = threadIdx.x; e < HIDDEN * XS; e += THREADS) {
    const int j = e / XS, k = e % XS;
    S.w1[j][k] = k < 9 ? w.w1[j * 9 + k] : (k == 9 ? w.b1[j] : 0.f);
    S.w3t[j][k] = k < 9 ? w.w3[k * HIDDEN + j] : 0.f;
    S.w1t[k][j] = k < 9 ? w.w1[j * 9 + k] : 0.f;
  }
  for (int e = threadIdx.x; e < HIDDEN * HIDDEN; e += THREADS) {
    const int j = e / HIDDEN, k = e % HIDDEN;
    const float v = w.w2[e];
    S.w2[j][k] = v;
    S.w2t[k][j] = v;
  }
  if (threadIdx.x < HIDDEN) S.b2[threadIdx.x] = w.b2[threadIdx.x];
  if (threadIdx.x < XS) S.b3[threadIdx.x] = threadIdx.x < 9 ? w.b3[threadIdx.x] : 0.f;
  const int group = threadIdx.x / TILE, t = threadIdx.x % TILE;
  Group &G = S.g[group];
#pragma unroll
  for (int k = 0; k < SMALL; ++k) G.small[k][t] = 0.f;
  __syncthreads();

  // matrix-product layouts: units c * 8 + ug of nodes r * 16 + ng; dL/dx components
  // c * 4 + xg of nodes r * 32 + ngx; dW2 entries (j0 + a, k0 + b); dW1, dW3 column j
  // over half of the nodes
  const int ug = t & 7, ng = t >> 3, xg = t & 3, ngx = t >> 2;
  const int j0 = 8 * (t >> 4), k0 = 4 * (t & 15), jc = t & (HIDDEN - 1), n0 = t & HIDDEN;
  const uint32_t bar = 1 + group;
  auto sync = [&]() { umma::named_barrier(bar, TILE); };
  float2 dw2[4][4];  // running sums of dW2: pairs of j x k
  clear(dw2);
  float db3[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) db3[i] = 0.f;

  const size_t plane = (size_t)nx * ny;
  const float omega = p.omega;
  for (long long tile = (long long)blockIdx.x * GROUPS + group; tile * TILE < nodes;
       tile += (long long)gridDim.x * GROUPS) {
    const long long n = tile * TILE + t;
    const bool active = n < nodes;
    int x = 0, y = 0;
    size_t base = 0;  // of this node's lattice
    float d[Q], pb[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) d[i] = pb[i] = 0.f;
    if (active) {
      const int b = (int)(n / (long long)plane);
      const long long r = n - b * (long long)plane;
      y = (int)(r / nx);
      x = (int)(r - (long long)y * nx);
      base = (size_t)b * Q * plane;
    }
    const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
    if (active) {
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const int xs = cx(i) == 0 ? x : (cx(i) == 1 ? xm : xp);
        const int ys = cy(i) == 0 ? y : (cy(i) == 1 ? ym : yp);
        d[i] = __ldg(state + base + i * plane + (size_t)ys * nx + xs);
        pb[i] = __ldg(lam_next + base + i * plane + (size_t)y * nx + x);
      }
    }
    float ob_b3 = 0.f;  // dL/do . b3
    {
      const Moments m = node_moments(d);
      float deq[Q], xin[Q], ob[Q];
      shifted_feq(m, deq);
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        xin[i] = active ? (d[i] - deq[i]) * m.inv_rho : 0.f;
        ob[i] = m.rho * omega * pb[i];
      }
      float4 *xr = reinterpret_cast<float4 *>(&G.x[t][0]);
      xr[0] = make_float4(xin[0], xin[1], xin[2], xin[3]);
      xr[1] = make_float4(xin[4], xin[5], xin[6], xin[7]);
      xr[2] = make_float4(xin[8], active ? 1.0f : 0.0f, 0.f, 0.f);
      project9(ob);  // dL/do = P^T dL/dohat, P symmetric
      float4 *orow = reinterpret_cast<float4 *>(&G.ob[t][0]);
      orow[0] = make_float4(ob[0], ob[1], ob[2], ob[3]);
      orow[1] = make_float4(ob[4], ob[5], ob[6], ob[7]);
      orow[2] = make_float4(ob[8], 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        db3[i] += ob[i];
        ob_b3 = fmaf(ob[i], S.b3[i], ob_b3);
      }
    }
    sync();
    // h1 = tanh(W1 x + b1), h2 = tanh(W2 h1 + b2) (one copy of the epilogue)
#pragma unroll 1
    for (int layer = 1; layer <= 2; ++layer) {
      float2 acc[8][8];
      clear(acc);
      if (layer == 1)
        dense_acc<8, 8, XS / 4, XS, XS>(&G.x[ng][0], 16, &S.w1[ug][0], 8, acc);
      else
        dense_acc<8, 8, HIDDEN / 4, HS, HS>(&G.h1[ng][0], 16, &S.w2[ug][0], 8, acc);
      float *dst = (layer == 1 ? &G.h1[ng][0] : &G.h2[ng][0]) + ug;
#pragma unroll
      for (int c = 0; c < 8; c += 2) {
        const float2 bias = layer == 1 ? make_float2(0.f, 0.f)
                                       : make_float2(S.b2[c * 8 + ug], S.b2[c * 8 + 8 + ug]);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const float2 h =
              tanh2(__fadd2_rn(make_float2(total(acc[r][c]), total(acc[r][c + 1])), bias));
          dst[r * 16 * HS + c * 8] = h.x;
          dst[r * 16 * HS + c * 8 + 8] = h.y;
        }
      }
      sync();
    }
    {  // dW3[i][jc] over nodes n0 .. n0 + 63
      float2 c[5];
#pragma unroll
      for (int i = 0; i < 5; ++i) c[i] = make_float2(0.f, 0.f);
#pragma unroll 4
      for (int k = 0; k < HIDDEN; ++k) {
        const float4 *o = reinterpret_cast<const float4 *>(&G.ob[n0 + k][0]);
        const float4 o0 = o[0], o1 = o[1];
        const float h = G.h2[n0 + k][jc], o8 = G.ob[n0 + k][8];
        const float2 hh = make_float2(h, h);
        c[0] = __ffma2_rn(make_float2(o0.x, o0.y), hh, c[0]);
        c[1] = __ffma2_rn(make_float2(o0.z, o0.w), hh, c[1]);
        c[2] = __ffma2_rn(make_float2(o1.x, o1.y), hh, c[2]);
        c[3] = __ffma2_rn(make_float2(o1.z, o1.w), hh, c[3]);
        c[4].x = fmaf(o8, h, c[4].x);
      }
#pragma unroll
      for (int i = 0; i < Q; ++i) G.small[10 + i][t] += i & 1 ? c[i / 2].y : c[i / 2].x;
    }
    sync();
    {  // dL/da2 and (dL/do W3) . h2
      float2 acc[8][8];
      clear(acc);
      dense_acc<8, 8, XS / 4, XS, XS>(&G.ob[ng][0], 16, &S.w3t[ug][0], 8, acc);
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        float s = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          float &e = G.h2[r * 16 + ng][c * 8 + ug];
          const float h = e, g = total(acc[r][c]);
          s = fmaf(g, h, s);
          e = g * (1.0f - h * h);
        }
        for (int off = 1; off < 8; off <<= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (ug == 0) G.dot[r * 16 + ng] = s;
      }
    }
    sync();
    {  // dW2 and db2
      float2 c[4][4];
      clear(c);
#pragma unroll 4
      for (int k = 0; k < TILE; ++k) {
        const float4 a0 = *reinterpret_cast<const float4 *>(&G.h2[k][j0]);
        const float4 a1 = *reinterpret_cast<const float4 *>(&G.h2[k][j0 + 4]);
        const float4 h = *reinterpret_cast<const float4 *>(&G.h1[k][k0]);
        const float2 aa[4] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w),
                              make_float2(a1.x, a1.y), make_float2(a1.z, a1.w)};
        const float hh[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int a = 0; a < 4; ++a)
            c[a][q] = __ffma2_rn(aa[a], make_float2(hh[q], hh[q]), c[a][q]);
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int q = 0; q < 4; ++q) dw2[a][q] = __fadd2_rn(dw2[a][q], c[a][q]);
      float s = 0.f;
#pragma unroll 8
      for (int k = 0; k < HIDDEN; ++k) s += G.h2[n0 + k][jc];
      G.small[19][t] += s;
    }
    {  // dL/da1
      float2 acc[8][8];
      clear(acc);
      dense_acc<8, 8, HIDDEN / 4, HS, HS>(&G.h2[ng][0], 16, &S.w2t[ug][0], 8, acc);
      sync();  // dL/da2 is read
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float h = G.h1[r * 16 + ng][c * 8 + ug];
          G.h2[r * 16 + ng][c * 8 + ug] = total(acc[r][c]) * (1.0f - h * h);
        }
    }
    sync();
    {  // [dW1 | db1][jc][k] over nodes n0 .. n0 + 63
      float2 c[5];
#pragma unroll
      for (int i = 0; i < 5; ++i) c[i] = make_float2(0.f, 0.f);
#pragma unroll 4
      for (int k = 0; k < HIDDEN; ++k) {
        const float4 *xr = reinterpret_cast<const float4 *>(&G.x[n0 + k][0]);
        const float4 x0 = xr[0], x1 = xr[1];
        const float2 x2 = *reinterpret_cast<const float2 *>(&G.x[n0 + k][8]);
        const float a = G.h2[n0 + k][jc];
        const float2 aa = make_float2(a, a);
        c[0] = __ffma2_rn(make_float2(x0.x, x0.y), aa, c[0]);
        c[1] = __ffma2_rn(make_float2(x0.z, x0.w), aa, c[1]);
        c[2] = __ffma2_rn(make_float2(x1.x, x1.y), aa, c[2]);
        c[3] = __ffma2_rn(make_float2(x1.z, x1.w), aa, c[3]);
        c[4] = __ffma2_rn(x2, aa, c[4]);
      }
#pragma unroll
      for (int i = 0; i < 10; ++i) G.small[i][t] += i & 1 ? c[i / 2].y : c[i / 2].x;
    }
    {  // dL/dx (dL/do is read)
      float2 acc[4][3];
      clear(acc);
      dense_acc<4, 3, HIDDEN / 4, HS, HS>(&G.h2[ngx][0], 32, &S.w1t[xg][0], 4, acc);
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) G.ob[r * 32 + ngx][c * 4 + xg] = total(acc[r][c]);
    }
    sync();
    if (active) {
      // post = d + omega (deq - d) + rho omega ohat + fext(rho, u), x = (f - feq)/rho
      const Moments m = node_moments(d);
      float deq[Q], fb[Q];
      shifted_feq(m, deq);
      float rhob = (G.dot[t] + ob_b3) * m.inv_rho, uxb = 0.f, uyb = 0.f;
      if (p.force) {
        // f_ext = feq(rho, u + a) - feq(rho, u), a = (fx/rho, 0): the differences
        // of the two sums, written without cancellation (s = 2 u_x + a_x), and
        // the rho-dependence of a
        const float fx = __ldg(p.force + y);
        const float ax = fx * m.inv_rho;
        const float sxs = 2.0f * m.ux + ax, uxs = m.ux + ax;
        const GMom q = weighted_moments(pb);
        const float sx1 =
            m.rho * (3.0f * q.gx + 9.0f * (uxs * q.gxx + m.uy * q.gxy) - 3.0f * uxs * q.g0);
        rhob += ax * (3.0f * q.gx + 4.5f * (sxs * q.gxx + 2.0f * m.uy * q.gxy) -
                      1.5f * sxs * q.g0) -
                ax * m.inv_rho * sx1;
        uxb += m.rho * ax * (9.0f * q.gxx - 3.0f * q.g0);
        uyb += m.rho * ax * 9.0f * q.gxy;
      }
      GMom q = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // moments of dL/dfeq
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const float xb = G.ob[t][i] * m.inv_rho;
        const float xin = (d[i] - deq[i]) * m.inv_rho;
        fb[i] = pb[i] * (1.0f - omega) + xb;
        gmom_add(q, i, pb[i] * omega - xb);
        rhob -= xb * xin;
      }
      float sr, sx, sy;
      feq_vjp(q, m.rho, m.ux, m.uy, sr, sx, sy);
      rhob += sr;
      uxb += sx;
      uyb += sy;
      // u = j / rho; rho = sum f, j = sum f c
      const float jxb = uxb * m.inv_rho, jyb = uyb * m.inv_rho;
      rhob -= (uxb * m.ux + uyb * m.uy) * m.inv_rho;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const float v = fb[i] + rhob + (float)cx(i) * jxb + (float)cy(i) * jyb;
        const int xs = cx(i) == 0 ? x : (cx(i) == 1 ? xm : xp);
        const int ys = cy(i) == 0 ? y : (cy(i) == 1 ? ym : yp);
        lam_out[base + i * plane + (size_t)ys * nx + xs] = v;  // lam_i(x - c_i)
      }
    }
  }
  // ---- each group's sums into its h1, then the groups' in order
  sync();
  float *sum = &G.h1[0][0];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      sum[OFF_W2 + (j0 + 2 * a) * HIDDEN + k0 + q] = dw2[a][q].x;
      sum[OFF_W2 + (j0 + 2 * a + 1) * HIDDEN + k0 + q] = dw2[a][q].y;
    }
  if (t < HIDDEN) {
#pragma unroll
    for (int k = 0; k < 10; ++k) {
      const float v = G.small[k][t] + G.small[k][t + HIDDEN];
      if (k < 9) sum[OFF_W1 + t * 9 + k] = v;
      else sum[OFF_B1 + t] = v;
    }
#pragma unroll
    for (int i = 0; i < Q; ++i)
      sum[OFF_W3 + i * HIDDEN + t] = G.small[10 + i][t] + G.small[10 + i][t + HIDDEN];
    sum[OFF_B2 + t] = G.small[19][t] + G.small[19][t + HIDDEN];
  }
  // db3: sums over the group's threads (per warp, then the four warps in order)
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    float v = db3[i];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((t & 31) == 0) G.dot[4 * i + (t >> 5)] = v;
  }
  sync();
  if (t < Q) sum[OFF_B3 + t] = (G.dot[4 * t] + G.dot[4 * t + 1]) + (G.dot[4 * t + 2] + G.dot[4 * t + 3]);
  __syncthreads();
  float *row = partials + (size_t)blockIdx.x * NPARAMS;
  const float *s0 = &S.g[0].h1[0][0], *s1 = &S.g[1].h1[0][0];
  for (int e = threadIdx.x; e < NPARAMS; e += THREADS) {
    const float v = s0[e] + s1[e];
    row[e] = accumulate ? row[e] + v : v;
  }
}

// dW[e] = sum over rows r (in order) of partials[r][e], FP64 accumulation.
__global__ void k_reduce_dw(const float *__restrict__ partials, int rows, float *__restrict__ dW) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= NPARAMS) return;
  double s = 0.0;
  for (int r = 0; r < rows; ++r) s += (double)partials[(size_t)r * NPARAMS + e];
  dW[e] = (float)s;
}

}  // namespace

int adjoint_blocks(const Grid &g, int sms) {
  const long long blocks = ((long long)g.nodes() + THREADS - 1) / THREADS;
  return (int)(blocks < sms ? blocks : sms);
}

cudaError_t launch_adjoint_step(const Grid &g, const float *state_n, const float *lam_next,
                                float *lam_out, const CollideParams &p, const MlpF32 &w,
                                float *dw_partials, int rows, int accumulate, cudaStream_t s) {
  const cudaError_t e = allow_smem(k_adjoint_step, sizeof(AdjSmem));
  if (e != cudaSuccess) return e;
  k_adjoint_step<<<rows, THREADS, sizeof(AdjSmem), s>>>(state_n, lam_next, lam_out, g.nx, g.ny,
                                                        (long long)g.nodes(), p, w, dw_partials,
                                                        accumulate);
  return cudaGetLastError();
}

cudaError_t launch_reduce_dw(const float *dw_partials, int rows, float *dW, cudaStream_t s) {
  k_reduce_dw<<<(NPARAMS + 255) / 256, 256, 0, s>>>(dw_partials, rows, dW);
  return cudaGetLastError();
}

}  // namespace lbm
