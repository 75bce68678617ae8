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

// tanh of two values.  |x| < 1: x + x u P(u), u = x^2, with the degree-6
// polynomial of least relative error there (Lawson-weighted least squares,
// 2^-28); otherwise 1 - 2 t / (1 + t) with t = e^{-2|x|} from the hardware's
// single-instruction power of two and reciprocal, which run beside the FMA pipe.
// The exponent y = -2 log2(e) |x| is rounded; its rounding error, which an FMA
// yields exactly, goes into t to first order.
// Errors in units of 2^-24 of tanh, root mean square / maximum over 4 M points
// per band, beside tanhf's (the maximum of a band varies by several per cent with
// its points):
//   |x| in  0 - 0.8      0.8 - 1      1 - 1.2      1.2 - 1.6    1.6 - 2      2 - 9
//   tanh2   0.45 / 1.27  0.44 / 1.30  0.46 / 1.88  0.37 / 1.40  0.31 / 0.86  0.29 / 0.65
//   tanhf   1.01 / 3.30  0.63 / 2.37  0.46 / 1.78  0.38 / 1.30  0.32 / 0.95  0.29 / 0.68
// About 14 issue slots per value against more than 20.  Without the correction
// and with a degree-5 polynomial up to 0.8 (11 slots; the FP32 step 3.5 % faster)
// it was 0.69 / 2.85 from 0.8 to 1 and up to 5 % above tanhf from there to 2.
__device__ __forceinline__ float2 tanh2(float2 x) {
  constexpr float P[7] = {-0.33333295583724976f, 0.13332344591617584f,   -0.05387980118393898f,
                          0.021486656740307808f, -0.007946106605231762f, 0.0023013644386082888f,
                          -0.0003584519727155566f};
  constexpr float K = 2.8853900817779268f, LN2 = 0.69314718055994531f;
  const float2 u = __fmul2_rn(x, x);
  float2 p = make_float2(P[6], P[6]);
#pragma unroll
  for (int k = 5; k >= 0; --k) p = __ffma2_rn(p, u, make_float2(P[k], P[k]));
  const float2 s = __ffma2_rn(x, __fmul2_rn(u, p), x);
  // (bounded, so that an infinite x makes no NaN; 1 - tanh(20) < 2^-25)
  const float2 a = make_float2(fminf(fabsf(x.x), 20.0f), fminf(fabsf(x.y), 20.0f));
  const float2 y = __fmul2_rn(a, make_float2(-K, -K));
  const float2 c = __ffma2_rn(a, make_float2(K, K), y);  // the exponent is y - c
  float2 t, r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(t.x) : "f"(y.x));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(t.y) : "f"(y.y));
  t = __ffma2_rn(t, __fmul2_rn(c, make_float2(-LN2, -LN2)), t);
  const float2 d = __fadd2_rn(t, make_float2(1.0f, 1.0f));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(d.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(d.y));
  const float2 l = __ffma2_rn(__fmul2_rn(t, r), make_float2(-2.0f, -2.0f), make_float2(1.0f, 1.0f));
  return make_float2(fabsf(x.x) >= 1.0f ? copysignf(l.x, x.x) : s.x,  // a NaN stays one
                     fabsf(x.y) >= 1.0f ? copysignf(l.y, x.y) : s.y);
}

}  // namespace f32
}  // namespace lbm
