// dense_f32.cuh -- FP32 building blocks of the 9 -> 64 -> 64 -> 9 network on the
// CUDA cores, for tiles of 128 nodes and 128 threads: matrix products in packed
// f32x2 arithmetic with operands in shared memory, and an accurate tanh.
//
// Operands are row-major [row][k] with a row stride that is 4 or 12 modulo 32
// floats, so that loads of consecutive rows are free of bank conflicts.  A
// thread sums R x C outputs, each with the sums over the even and the odd inputs
// in one packed accumulator (adjacent inputs pair up without any move), and per
// two inputs reads R + C 8-byte words for R C packed FMAs.
#pragma once
#include <cuda_runtime.h>

#include "lattice.cuh"

namespace lbm {
namespace f32 {

constexpr int TILE = 128;  // nodes per tile and threads that work on it
constexpr int HS = 68;     // row stride of the hidden vectors and of 64-wide weights
constexpr int XS = 12;     // row stride of the 9-vectors (with bias column)

// acc[r][c] += (even, odd) partial sums of A[a0 + r AR] . B[b0 + c BR] over 4 K4
// inputs; a, b point at rows a0 and b0.  Not unrolled further: the body is 160
// instructions, and a loop twice as long misses the instruction cache (the FP32
// step then takes 50 % more).  16-byte loads with four inputs per body and
// loads one body ahead were 4-5 % slower.
template <int R, int C, int K4, int AS, int BS>
__device__ __forceinline__ void dense_acc(const float *a, int a_step, const float *b, int b_step,
                                          float2 (&acc)[R][C]) {
#pragma unroll 2
  for (int k = 0; k < 2 * K4; ++k) {
    float2 av[R];
#pragma unroll
    for (int r = 0; r < R; ++r) av[r] = *reinterpret_cast<const float2 *>(a + r * a_step * AS + 2 * k);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const float2 bv = *reinterpret_cast<const float2 *>(b + c * b_step * BS + 2 * k);
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r][c] = __ffma2_rn(av[r], bv, acc[r][c]);
    }
  }
}
template <int R, int C>
__device__ __forceinline__ void clear(float2 (&acc)[R][C]) {
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < C; ++c) acc[r][c] = make_float2(0.f, 0.f);
}
__device__ __forceinline__ float total(float2 s) { return s.x + s.y; }

// tanh of two values.  |x| < 0.8: x + x u P(u), u = x^2, with the degree-5
// polynomial of least relative error there (Lawson-weighted least squares,
// 2^-28); otherwise 1 - 2 t / (1 + t) with t = e^{-2|x|} from the hardware's
// single-instruction power of two and reciprocal, which run beside the FMA pipe.
// About 11 issue slots per value against more than 20 of tanhf, with its
// accuracy (root mean square and maximum error over [-9, 9] no larger; the
// measured figures stand at k_step_mlp_f32).
__device__ __forceinline__ float2 tanh2(float2 x) {
  constexpr float P0 = -0.33333298563957214f, P1 = 0.13332220911979675f,
                  P2 = -0.05385233089327812f, P3 = 0.02130299061536789f,
                  P4 = -0.0074095577001571655f, P5 = 0.0015847564209252596f;
  const float2 u = __fmul2_rn(x, x);
  float2 p = __ffma2_rn(make_float2(P5, P5), u, make_float2(P4, P4));
  p = __ffma2_rn(p, u, make_float2(P3, P3));
  p = __ffma2_rn(p, u, make_float2(P2, P2));
  p = __ffma2_rn(p, u, make_float2(P1, P1));
  p = __ffma2_rn(p, u, make_float2(P0, P0));
  const float2 s = __ffma2_rn(x, __fmul2_rn(u, p), x);
  float2 t, r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(t.x) : "f"(-2.8853900817779268f * fabsf(x.x)));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(t.y) : "f"(-2.8853900817779268f * fabsf(x.y)));
  const float2 d = __fadd2_rn(t, make_float2(1.0f, 1.0f));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(d.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(d.y));
  const float2 l = __ffma2_rn(__fmul2_rn(t, r), make_float2(-2.0f, -2.0f), make_float2(1.0f, 1.0f));
  return make_float2(fabsf(x.x) < 0.8f ? s.x : copysignf(l.x, x.x),
                     fabsf(x.y) < 0.8f ? s.y : copysignf(l.y, x.y));
}

}  // namespace f32
}  // namespace lbm
