// diag.cu -- flow diagnostics of the turbulence statistics the paper reports:
// longitudinal velocity structure functions (SI section 3) and the shell-
// averaged kinetic energy spectrum (main text, energy spectra).
//
// Structure functions: S^p(r) = < [(u(x + r e) - u(x)) . e]^p >, p = 1..6,
// r = 1..rmax, averaged over every node and the two lattice directions
// e = x^, y^ (periodic).  For rmax <= 256: strips of 32 lines staged in shared
// memory with an rmax halo, one thread per separation; otherwise one block per
// (r, chunk of rows).  Either way per-thread FP32 sums over at most 32 nodes are
// flushed into FP64 (or FP32-triple) accumulators and per-block FP64 partials are
// added in a fixed order, so results are reproducible.
//
// Energy spectrum: E(k) = 1/2 sum_{round(|k'|) = k} |u_hat(k')|^2 / N^2 for the
// unnormalised 2D DFT (N = nx ny), averaged over the batch, so that the sum
// over all shells is <|u|^2>/2.  The DFT is a cuFFT R2C call; the binning is
// deterministic: shell s collects, in each ky row, the contiguous range of
// kx >= 0 with s^2 - s + 1 <= kx^2 + ky^2 <= s^2 + s, summed by one thread,
// with weight 2 for the kx that stand for their conjugate -kx.
#include <cstdint>
#include <cufft.h>

#include "kernels.h"

namespace lbm {
namespace {

constexpr int SF_THREADS = 256;

__global__ void __launch_bounds__(SF_THREADS)
    k_structure_partials(const float *__restrict__ ux, const float *__restrict__ uy, int nx,
                         int ny, int batch, int rows_per_block, double *__restrict__ part) {
  const int r = blockIdx.x + 1;
  const int chunk = blockIdx.y;
  const int total_rows = ny * batch;
  const int row0 = chunk * rows_per_block;
  const int row1 = min(row0 + rows_per_block, total_rows);
  double acc[6] = {0, 0, 0, 0, 0, 0};
  float facc[6] = {0, 0, 0, 0, 0, 0};
  int pending = 0;
  const size_t N = (size_t)nx * ny;
  for (int row = row0; row < row1; ++row) {
    const int b = row / ny, y = row % ny;
    const int yr = y + r >= ny ? (y + r) % ny : y + r;
    const float *uxr = ux + (size_t)b * N + (size_t)y * nx;
    const float *uyr = uy + (size_t)b * N + (size_t)y * nx;
    const float *uyr2 = uy + (size_t)b * N + (size_t)yr * nx;
    for (int x = threadIdx.x; x < nx; x += SF_THREADS) {
      const int xr = x + r >= nx ? (x + r) % nx : x + r;
      const float dx = uxr[xr] - uxr[x];
      const float dy = uyr2[x] - uyr[x];
      float px = dx, py = dy;
#pragma unroll
      for (int p = 0; p < 6; ++p) {
        facc[p] += px + py;
        px *= dx;
        py *= dy;
      }
      if (++pending == 32) {
#pragma unroll
        for (int p = 0; p < 6; ++p) {
          acc[p] += (double)facc[p];
          facc[p] = 0.f;
        }
        pending = 0;
      }
    }
  }
#pragma unroll
  for (int p = 0; p < 6; ++p) acc[p] += (double)facc[p];
  __shared__ double red[6][SF_THREADS];
#pragma unroll
  for (int p = 0; p < 6; ++p) red[p][threadIdx.x] = acc[p];
  __syncthreads();
  for (int w = SF_THREADS / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w)
#pragma unroll
      for (int p = 0; p < 6; ++p) red[p][threadIdx.x] += red[p][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < 6)
    part[((size_t)(r - 1) * gridDim.y + chunk) * 6 + threadIdx.x] = red[threadIdx.x][0];
}

// Tiled form for rmax <= SFT_R (the usual case): one pass over the field per
// direction instead of one per separation.  A block stages 32 rows (for the x
// increments) or 32 columns (y) over h positions along the increments and the
// next rmax ones (periodic) in shared memory; thread r - 1 owns separation r.
// Two nodes at a time in packed f32x2: two rows for the x increments, stored as
// [x][row] so that 16-byte loads give four rows (a stride of 36 floats keeps
// them free of bank conflicts); two positions for the y increments, stored as
// [column][y].  Nine FMA-pipe operations per increment for its six powers
// bound the kernel.  Each lane sums 32 terms, adjacent in x, in FP32 (S^1 is the
// rounding left of a sum that cancels, so the order is part of the result)
// before they go into its running sum, three FP32 numbers kept by error-free
// additions (more than the 53 bits of a double): FP64 additions, at 1/64 of the
// FP32 rate, took as long as all the rest.
// Measured (GB300, 1024^2, r <= 256, E(k) and S^p(r) together): 0.36 ms, 1.04
// before; 0.34 ms with pairs of FP32 numbers (48 bits).
constexpr int SFT_R = 256;    // largest separation
constexpr int SF_LINES = 32;
constexpr int SF_STRIDE = SF_LINES + 4;  // of a position of the x increments
constexpr int SF_MOST_BLOCKS = 4096;

// (h, l, m) += f: every rounding error of h caught in l and every one of l in m
// (Knuth's two-sum), per lane.
__device__ __forceinline__ float2 two_sum(float2 &a, float2 f) {
  const float2 m1 = make_float2(-1.f, -1.f);
  const float2 s = __fadd2_rn(a, f), b = __ffma2_rn(a, m1, s);
  const float2 e = __fadd2_rn(__ffma2_rn(__ffma2_rn(b, m1, s), m1, a), __ffma2_rn(b, m1, f));
  a = s;
  return e;
}
__device__ __forceinline__ void sum3_add(float2 &h, float2 &l, float2 &m, float2 f) {
  m = __fadd2_rn(m, two_sum(l, two_sum(h, f)));
}

// a modulo n, n <= a < 2 n in the usual case
__device__ __forceinline__ int periodic(int a, int n) {
  a -= a >= n ? n : 0;
  return a < n ? a : a % n;
}

struct SfShape {
  int h;             // positions per block
  int bx, by;        // blocks of the x and of the y increments
  int segs_x, segs_y;  // blocks along the axis
};

__global__ void __launch_bounds__(SFT_R, 3)
    k_sf_strips(const float *__restrict__ ux, const float *__restrict__ uy, int nx, int ny,
                int batch, int rmax, SfShape sh, double *__restrict__ part) {
  extern __shared__ __align__(16) float strip[];  // (h + rmax) positions of 32 lines
  const bool along_x = (int)blockIdx.x < sh.bx;
  const int ystride = (sh.h + rmax + 2) / 4 * 4 + 2;  // even: aligned pairs; 2-way when staged
  const int rt = (rmax + 31) / 32 * 32;  // threads per slice; slices share the positions
  const int slices = blockDim.x / rt, slice = threadIdx.x / rt, r = threadIdx.x % rt + 1;
  int h;
  if (along_x) {
    // 32 rows of the flattened batch, positions along x
    const int p0 = blockIdx.x % sh.segs_x * sh.h, l0 = blockIdx.x / sh.segs_x * SF_LINES;
    h = min(sh.h, nx - p0);
    const int lw = min(SF_LINES, ny * batch - l0);
    for (int l = threadIdx.x / 32; l < SF_LINES; l += blockDim.x / 32)
      for (int j = threadIdx.x % 32; j < h + rmax; j += 32)
        strip[j * SF_STRIDE + l] = l < lw ? ux[(size_t)(l0 + l) * nx + periodic(p0 + j, nx)] : 0.f;
  } else {
    // 32 columns of one lattice, positions along y
    const int blk = blockIdx.x - sh.bx, strips = (nx + SF_LINES - 1) / SF_LINES;
    const int l0 = blk % strips * SF_LINES, q = blk / strips;
    const int p0 = q % sh.segs_y * sh.h;
    h = min(sh.h, ny - p0);
    const int lw = min(SF_LINES, nx - l0), l = threadIdx.x % 32;
    const float *u = uy + (size_t)(q / sh.segs_y) * nx * ny + l0 + l;
    for (int j = threadIdx.x / 32; j < h + rmax; j += blockDim.x / 32)
      strip[l * ystride + j] = l < lw ? u[(size_t)periodic(p0 + j, ny) * nx] : 0.f;
  }
  __syncthreads();
  float2 hi[6], lo[6], lo2[6];
#pragma unroll
  for (int p = 0; p < 6; ++p) hi[p] = lo[p] = lo2[p] = make_float2(0.f, 0.f);
  const float2 m1 = make_float2(-1.f, -1.f);
  auto add = [](float2 (&f)[6], float2 d) {
    const float2 d2 = __fmul2_rn(d, d), d3 = __fmul2_rn(d2, d);
    f[0] = __fadd2_rn(f[0], d);
    f[1] = __fadd2_rn(f[1], d2);
    f[2] = __fadd2_rn(f[2], d3);
    f[3] = __ffma2_rn(d2, d2, f[3]);
    f[4] = __ffma2_rn(d2, d3, f[4]);
    f[5] = __ffma2_rn(d3, d3, f[5]);
  };
  if (slice < slices && r <= rmax) {
    if (along_x) {
      // runs of 32 positions of four rows
      for (int k = slice; k < (h + 31) / 32 * (SF_LINES / 4); k += slices) {
        const int j0 = k / (SF_LINES / 4) * 32, n = min(32, h - j0);
        const float *s0 = strip + j0 * SF_STRIDE + 4 * (k % (SF_LINES / 4));
        const float *s1 = s0 + r * SF_STRIDE;
        float2 f[2][6];
#pragma unroll
        for (int p = 0; p < 6; ++p) f[0][p] = f[1][p] = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int j = 0; j < n; ++j) {
          const float4 a = *reinterpret_cast<const float4 *>(s1 + j * SF_STRIDE);
          const float4 b = *reinterpret_cast<const float4 *>(s0 + j * SF_STRIDE);
          add(f[0], __ffma2_rn(make_float2(b.x, b.y), m1, make_float2(a.x, a.y)));
          add(f[1], __ffma2_rn(make_float2(b.z, b.w), m1, make_float2(a.z, a.w)));
        }
#pragma unroll
        for (int p = 0; p < 6; ++p) {
          sum3_add(hi[p], lo[p], lo2[p], f[0][p]);
          sum3_add(hi[p], lo[p], lo2[p], f[1][p]);
        }
      }
    } else {
      // 32 columns of two positions
      for (int j = 2 * slice; j < h; j += 2 * slices) {
        const float *s0 = strip + j, *s1 = s0 + r;
        const bool two = j + 1 < h;
        float2 f[6];
#pragma unroll
        for (int p = 0; p < 6; ++p) f[p] = make_float2(0.f, 0.f);
#pragma unroll 8
        for (int c = 0; c < SF_LINES; ++c) {
          float2 d = __ffma2_rn(*reinterpret_cast<const float2 *>(s0 + c * ystride), m1,
                                make_float2(s1[c * ystride], s1[c * ystride + 1]));
          if (!two) d.y = 0.f;
          add(f, d);
        }
#pragma unroll
        for (int p = 0; p < 6; ++p) sum3_add(hi[p], lo[p], lo2[p], f[p]);
      }
    }
  }
  double acc[6];
  bool finite = true;
#pragma unroll
  for (int p = 0; p < 6; ++p) {
    acc[p] = ((double)hi[p].x + (double)hi[p].y) +
             (((double)lo[p].x + (double)lo[p].y) + ((double)lo2[p].x + (double)lo2[p].y));
    finite &= isfinite(acc[p]);
  }
  if (!finite && slice < slices && r <= rmax) {
    // a blown-up field: the FP32 running sums may overflow where FP64 ones do
    // not, and two-sum turns an infinity into a NaN; add up in FP64 instead
#pragma unroll
    for (int p = 0; p < 6; ++p) acc[p] = 0.0;
    const int sp = along_x ? SF_STRIDE : 1, sl = along_x ? 1 : ystride;
    for (int j = 0; j < h; ++j) {
      for (int l = 0; l < SF_LINES; ++l) {
        // the nodes this slice took above
        if ((along_x ? j / 32 * (SF_LINES / 4) + l / 4 : j / 2) % slices != slice) continue;
        const float d = strip[(j + r) * sp + l * sl] - strip[j * sp + l * sl];
        float q = d;
        for (int p = 0; p < 6; ++p, q *= d) acc[p] += (double)q;
      }
    }
  }
  // slices in order, then one row of 6 x rmax partial sums per block
  if (slices > 1) {
    __syncthreads();  // the strip is read; its space takes the slices' sums
    double *red = reinterpret_cast<double *>(strip);  // [slices][6][rt]
    if (slice < slices)
#pragma unroll
      for (int p = 0; p < 6; ++p) red[(slice * 6 + p) * rt + r - 1] = acc[p];
    __syncthreads();
    if (slice == 0)
      for (int k = 1; k < slices; ++k)
#pragma unroll
        for (int p = 0; p < 6; ++p) acc[p] += red[(k * 6 + p) * rt + r - 1];
  }
  if (slice == 0 && r <= rmax)
#pragma unroll
    for (int p = 0; p < 6; ++p) part[((size_t)blockIdx.x * 6 + p) * rmax + r - 1] = acc[p];
}

// out[e] = scale * sum over k (in a fixed order) of rows[k][e]: 32 columns per
// block, the rows in 32 interleaved slices.
constexpr int SUM_SLICES = 32;
__global__ void __launch_bounds__(32 * SUM_SLICES)
    k_sum_rows(const double *__restrict__ rows, int n, int width, double scale,
               double *__restrict__ out) {
  __shared__ double red[SUM_SLICES][33];
  const int lane = threadIdx.x % 32, slice = threadIdx.x / 32;
  const int e = blockIdx.x * 32 + lane;
  double s = 0.0;
  if (e < width)
#pragma unroll 4
    for (int k = slice; k < n; k += SUM_SLICES) s += rows[(size_t)k * width + e];
  red[slice][lane] = s;
  __syncthreads();
  if (slice == 0 && e < width) {
    for (int k = 1; k < SUM_SLICES; ++k) s += red[k][lane];
    out[e] = s * scale;
  }
}

SfShape sf_shape(const Grid &g) {
  SfShape s;
  const long long rows = ((long long)g.ny * g.batch + SF_LINES - 1) / SF_LINES;
  const long long strips = (long long)((g.nx + SF_LINES - 1) / SF_LINES) * g.batch;
  // 32 positions per block (1,024 blocks per direction at 1024^2), up to 256
  // while that leaves more than SF_MOST_BLOCKS rows of partial sums
  for (s.h = 32;; s.h *= 2) {
    s.segs_x = (g.nx + s.h - 1) / s.h;
    s.segs_y = (g.ny + s.h - 1) / s.h;
    const long long bx = rows * s.segs_x, by = strips * s.segs_y;
    if (s.h == 256 || bx + by <= SF_MOST_BLOCKS) {
      s.bx = bx + by <= 0x7fffffffLL ? (int)bx : 0;
      s.by = bx + by <= 0x7fffffffLL ? (int)by : 0;
      return s;
    }
  }
}

// S[p][r] = sum over chunks (in order) / (2 B N)
__global__ void k_structure_final(const double *__restrict__ part, int rmax, int chunks,
                                  double inv_count, double *__restrict__ S) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 6 * rmax) return;
  const int p = e / rmax, r = e % rmax;
  double s = 0.0;
  for (int c = 0; c < chunks; ++c) s += part[((size_t)r * chunks + c) * 6 + p];
  S[e] = s * inv_count;
}

__device__ __forceinline__ long long isqrt_floor(long long v) {
  if (v <= 0) return 0;
  if (v < 1 << 24) {  // in single precision (FP64 roots took half of k_spectrum_rows)
    const int w = (int)v;
    int s = (int)sqrtf((float)w);
    while (s * s > w) --s;
    while ((s + 1) * (s + 1) <= w) ++s;
    return s;
  }
  long long s = (long long)sqrt((double)v);
  while (s * s > v) --s;
  while ((s + 1) * (s + 1) <= v) ++s;
  return s;
}

// One thread per (ky row j, shell s): sum of the weighted |u_hat|^2 of the row's
// kx range of shell s, for both velocity components and every lattice.
__global__ void k_spectrum_rows(const cufftComplex *__restrict__ uh, int nx, int ny, int batch,
                                int kmax, double *__restrict__ rowpart) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  if (s > kmax) return;
  const int nxh = nx / 2 + 1;
  const long long ky = j < (ny + 1) / 2 ? j : j - ny;
  const long long lo2 = s == 0 ? 0 : (long long)s * s - s + 1, hi2 = (long long)s * s + s;
  const long long ky2 = ky * ky;
  double acc = 0.0;
  if (hi2 >= ky2) {
    const long long a = lo2 - ky2;
    long long kx_lo = a <= 0 ? 0 : isqrt_floor(a - 1) + 1;  // smallest kx with kx^2 >= a
    long long kx_hi = isqrt_floor(hi2 - ky2);
    if (kx_hi > nxh - 1) kx_hi = nxh - 1;
    for (long long kx = kx_lo; kx <= kx_hi; ++kx) {
      const double wgt = (kx == 0 || (nx % 2 == 0 && kx == nx / 2)) ? 1.0 : 2.0;
      for (int c = 0; c < 2 * batch; ++c) {
        const cufftComplex z = uh[((size_t)c * ny + j) * nxh + kx];
        acc += wgt * ((double)z.x * z.x + (double)z.y * z.y);
      }
    }
  }
  rowpart[(size_t)j * (kmax + 1) + s] = acc;
}

}  // namespace

// Positions of x or y increments, or the slices' sums (6 doubles per thread).
static size_t sf_smem(int h, int rmax) {
  const size_t n = sizeof(float) * (size_t)(h + rmax + 3) * SF_STRIDE;
  return n > sizeof(double) * 6 * SFT_R ? n : sizeof(double) * 6 * SFT_R;
}

// The tiled form applies for rmax <= SFT_R and grids within its launch limits.
static bool sf_tiled(const Grid &g, int rmax) { return rmax <= SFT_R && sf_shape(g).bx > 0; }

size_t structure_partials_doubles(const Grid &g, int rmax) {
  if (sf_tiled(g, rmax)) {
    const SfShape s = sf_shape(g);
    return (size_t)(s.bx + s.by) * rmax * 6;
  }
  const int rows = g.ny * g.batch;
  const int rpb = 8;
  const int chunks = (rows + rpb - 1) / rpb;
  return (size_t)rmax * chunks * 6;
}

cudaError_t launch_structure_functions(const Grid &g, const float *ux, const float *uy, int rmax,
                                       double *part, double *S, cudaStream_t s) {
  if (sf_tiled(g, rmax)) {
    const SfShape sh = sf_shape(g);
    cudaError_t e = allow_smem(k_sf_strips, sf_smem(256, SFT_R));  // the largest
    if (e != cudaSuccess) return e;
    k_sf_strips<<<sh.bx + sh.by, SFT_R, sf_smem(sh.h, rmax), s>>>(ux, uy, g.nx, g.ny, g.batch,
                                                                     rmax, sh, part);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_sum_rows<<<(6 * rmax + 31) / 32, 32 * SUM_SLICES, 0, s>>>(
        part, sh.bx + sh.by, 6 * rmax, 1.0 / (2.0 * (double)g.nodes()), S);
    return cudaGetLastError();
  }
  const int rows = g.ny * g.batch;
  const int rpb = 8;
  const int chunks = (rows + rpb - 1) / rpb;
  if (chunks > 65535) return cudaErrorInvalidValue;
  k_structure_partials<<<dim3(rmax, chunks), SF_THREADS, 0, s>>>(ux, uy, g.nx, g.ny, g.batch, rpb,
                                                                  part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_structure_final<<<(6 * rmax + 255) / 256, 256, 0, s>>>(part, rmax, chunks,
                                                           1.0 / (2.0 * (double)g.nodes()), S);
  return cudaGetLastError();
}

size_t spectrum_rowpart_doubles(const Grid &g, int kmax) { return (size_t)g.ny * (kmax + 1); }

// u: [2B][ny][nx] real (ux of every lattice, then uy); uh: [2B][ny][nx/2+1].
cudaError_t launch_energy_spectrum(const Grid &g, float *u, void *uh, void **plan_io, int kmax,
                                   double *rowpart, double *E, cudaStream_t s) {
  cufftHandle plan;
  if (!*plan_io) {
    int n[2] = {g.ny, g.nx};
    if (cufftPlanMany(&plan, 2, n, nullptr, 1, g.ny * g.nx, nullptr, 1, g.ny * (g.nx / 2 + 1),
                      CUFFT_R2C, 2 * g.batch) != CUFFT_SUCCESS)
      return cudaErrorUnknown;
    *plan_io = reinterpret_cast<void *>(static_cast<uintptr_t>(plan) + 1);
  }
  plan = static_cast<cufftHandle>(reinterpret_cast<uintptr_t>(*plan_io) - 1);
  if (cufftSetStream(plan, s) != CUFFT_SUCCESS) return cudaErrorUnknown;
  if (cufftExecR2C(plan, u, static_cast<cufftComplex *>(uh)) != CUFFT_SUCCESS)
    return cudaErrorUnknown;
  dim3 grid((kmax + 1 + 127) / 128, g.ny);
  k_spectrum_rows<<<grid, 128, 0, s>>>(static_cast<const cufftComplex *>(uh), g.nx, g.ny,
                                       g.batch, kmax, rowpart);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const double N = (double)g.nx * g.ny;
  k_sum_rows<<<(kmax + 32) / 32, 32 * SUM_SLICES, 0, s>>>(rowpart, g.ny, kmax + 1,
                                                         0.5 / (N * N * g.batch), E);
  return cudaGetLastError();
}

void destroy_spectrum_plan(void *plan_io) {
  if (plan_io) cufftDestroy(static_cast<cufftHandle>(reinterpret_cast<uintptr_t>(plan_io) - 1));
}

}  // namespace lbm
