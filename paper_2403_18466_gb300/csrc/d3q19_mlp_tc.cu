// d3q19_mlp_tc.cu -- the paper's learned collision on D3Q19 with its network
// (19 -> 300 -> 300 -> 100 -> 19, LeakyReLU, conservation layer with kappa
// denominators 19 and 10) on the 5th-generation tensor cores: tcgen05 MMAs with
// BF16 operands and FP32 accumulation in tensor memory, fused with the pull-
// stream, the BGK update and the EDM forcing (populations stay FP32).
//
// Per node: x = (f - feq)/rho; h1 = lrelu(W1 x + b1); h2 = lrelu(W2 h1 + b2);
// h3 = lrelu(W3 h2 + b3); o = W4 h3 + b4; f' = f + (feq - f)/tau + (rho/tau) P o + f_ext.
//
// GEMMs per tile of M = 128 nodes, biases folded in as a constant-1 operand
// column:
//   L1  [128 x  32] x [ 32 x 304]   K = 19 inputs + 1 + 12 zeros; N = 300 + 4 zero rows
//   L2  [128 x 304] x [304 x 304]   K = 300 + 1 + 3 zeros
//   L3  [128 x 304] x [304 x 112]   N = 100 + 12 zero rows
//   L4  [128 x 112] x [112 x  32]   K = 100 + 1 + 11 zeros; N = 19 + 13 zero rows
// A tile is 128 consecutive nodes of the flattened lattice (rows, planes and
// lattices of a batch follow one another), so that narrow lattices fill it.
//
// A cluster of two CTAs works on two tiles at a time (cta_group::2, M = 256:
// each CTA's tensor memory holds its own tile's operands and accumulators, and
// each CTA's shared memory half of the rows of every weight matrix).  Half of
// all the weights is 140 KB, so they stay resident for the whole launch; one
// CTA alone would have to stream W2 (185 KB) again for every tile.
//
// N = 304 exceeds one MMA: L1 and L2 run as two passes, columns 0..159 and
// 160..303.  The A operands (x and the activations, as bf16 pairs) live in
// tensor memory next to the accumulators: the epilogue reads an accumulator
// row with tcgen05.ld and writes the activation row back with tcgen05.st.
// Columns of the tensor memory:
//     0..303  accumulator of L1 and L2; h2 replaces L2's in place
//   304..455  h1; then L3's accumulator (304..415), where h3 replaces it
//   456..487  layer-4 output          488..503  x
// h1 takes the K steps' columns in an order (H1_RUNS) in which the lower half
// avoids those h3 of the previous tile still occupies.
//
// What overlaps: L2's first pass starts when the lower half of h1 is written;
// the lower half of h2 is written while the second pass runs and the upper
// half while L3 consumes the lower one; the next tile's x, the final update of
// the previous tile and the pulls of the next one run beside all of that.
//
// What bounds it: the MMAs cost ~95 cycles each (N = 160 is at the tensor rate,
// N = 112 and 32 below it), 68 per tile; the rest of a tile's ~9.6 k cycles is
// the hop from L3 over L1 to L2 (a commit reaches its waiters ~700 cycles after
// the last MMA) and the drains, which share the tensor memory with the MMAs.
// Measured (GB300): 4.0 G nodes/s at 256^3 (1,020 TFLOP/s), 3.9 at 128^3, 3.49 at
// 64^3, where one CTA per tile of a row with W2 streamed ran at 2.74, 2.68 and
// 1.29 G nodes/s.
//
// Roles in a CTA of 480 threads (one CTA per SM, a cluster persistent over a
// contiguous range of tile pairs):
//   warps 0-3, 4-7 (WG0, WG1)  the epilogues, each half of the columns of each part
//   warps 8-11     (WG2)       node work: pulls, the layer-1 operand, the final
//                              update (conservation layer, BGK, force) and store
//   warps 12-14                MMA issue for both CTAs (one thread each of CTA 0)
// Hand-offs are mbarriers: the issuers' (x and A operands ready, output read;
// one arrival per warp of both CTAs, at CTA 0) and the MMA commits', which
// arrive in both CTAs.  Every wait is bounded; on a time-out the role records
// it in both CTAs, all roles leave their loops, MMAs in flight are drained
// with a bounded wait, the tensor memory is freed and the timeout flag is set.
#include <cuda_bf16.h>

#include "d3q19.cuh"
#include "kernels3d.h"
#include "umma.cuh"

namespace lbm {
namespace d3 {
namespace {

using namespace umma;

constexpr int KX = 32;     // layer-1 K
constexpr int NH = 304;    // padded hidden width (rows of W1, W2 as B operands)
constexpr int NLO = 160, NHI = NH - NLO;  // the two passes of L1 and L2
constexpr int KH = 304;    // K of layers 2 and 3
constexpr int N3 = 112;    // rows of W3
constexpr int K4 = 112;    // K of layer 4
constexpr int N4 = 32;     // rows of W4
// one CTA's half of the weights: of each pass, half of the rows
constexpr int R_LO = NLO / 2, R_HI = NHI / 2, R_H = R_LO + R_HI;
constexpr int W1_BYTES = R_H * KX * 2;
constexpr int W2_BYTES = R_H * KH * 2;
constexpr int W3_BYTES = N3 / 2 * KH * 2;
constexpr int W4_BYTES = N4 / 2 * K4 * 2;
constexpr int G_W1 = 0, G_W2 = G_W1 + W1_BYTES, G_W3 = G_W2 + W2_BYTES, G_W4 = G_W3 + W3_BYTES;
constexpr int G_BYTES = G_W4 + W4_BYTES;  // 139,776 per CTA of the pair
static_assert(R_LO % 8 == 0 && R_HI % 8 == 0 && G_BYTES % 16 == 0, "operand halves");

// tensor-memory columns
constexpr uint32_t TM_P = 0, TM_A = 304, TM_OUT = 456, TM_X = 488;
// First column of K step s (16 inputs, 8 columns) of h1, h2 and h3, as packed
// tables of 6-bit entries (columns / 8), so that the issue loops stay small.
struct ColTable {
  uint64_t lo, hi;  // K steps 0..9, 10..18
  __host__ __device__ constexpr uint32_t operator()(int s) const {
    return 8u * (uint32_t)(((s < 10 ? lo : hi) >> (6 * (s < 10 ? s : s - 10))) & 63u);
  }
};
struct Run {
  int k0, n, col;  // K steps k0 .. k0 + n - 1 at col, col + 8, ...
};
template <int N>
constexpr ColTable make_table(const Run (&runs)[N]) {
  ColTable t{0, 0};
  for (int r = 0; r < N; ++r)
    for (int i = 0; i < runs[r].n; ++i) {
      const int s = runs[r].k0 + i;
      const uint64_t v = (uint64_t)(runs[r].col / 8 + i);
      if (s < 10) t.lo |= v << (6 * s);
      else t.hi |= v << (6 * (s - 10));
    }
  return t;
}
// the runs of the epilogues' parts: (WG0 | WG1) x (lower | upper), two runs each
constexpr Run H1_RUNS[8] = {{0, 4, 336},  {4, 1, 416},  {5, 3, 392},  {8, 2, 424},
                            {10, 4, 304}, {14, 1, 440}, {15, 3, 368}, {18, 1, 448}};
constexpr Run H2_RUNS[4] = {{0, 5, 0}, {5, 5, 80}, {10, 5, 160}, {15, 4, 240}};
constexpr Run H3_RUNS[2] = {{0, 4, 304}, {4, 3, 368}};
constexpr ColTable T1 = make_table(H1_RUNS), T2 = make_table(H2_RUNS), T3 = make_table(H3_RUNS);
__device__ __forceinline__ ColTable col_h1() { return ColTable{T1.lo, T1.hi}; }
__device__ __forceinline__ ColTable col_h2() { return ColTable{T2.lo, T2.hi}; }
__device__ __forceinline__ ColTable col_h3() { return ColTable{T3.lo, T3.hi}; }

constexpr int TILE = 128;
constexpr int NODE_WARP = 8, MMA_WARP = 12;
constexpr int THREADS = 32 * (MMA_WARP + 3);
// bounded waits: polls, each suspended for at most POLL_NS (1 s in all)
constexpr uint32_t WAIT_LIMIT = 1u << 18, POLL_NS = 4000;

struct __align__(1024) Smem {
  unsigned char w[G_BYTES];
  // the issuers' barriers (those of CTA 0 are used): x, halves of h1 and h2, h3, output read
  unsigned long long bx, b1lo, b1hi, b2lo, b2hi, b3, bo;
  // MMA commits (both CTAs'): L1 and L2 (two passes each), L3, L4
  unsigned long long c1a, c1b, c2a, c2b, c3, c4;
  unsigned long long wload, drain[3];
  uint32_t taddr;
  int err;
};
constexpr size_t SMEM_BYTES = sizeof(Smem) + 1024;
static_assert(SMEM_BYTES <= 232448, "shared memory layout too large");

// ---- helpers ------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
// Shared-memory address of the same variable in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_cta(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Arrivals and waits order tensor-memory accesses only (through the tcgen05
// fences around them), no generic memory, so they need no cluster-wide
// release or acquire: those cost ~1,000 and ~400 cycles each.
__device__ __forceinline__ void arrive_cluster(uint32_t mapped) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(mapped) : "memory");
}
__device__ __forceinline__ bool try_wait(uint32_t bar, uint32_t parity) {
  return mbar_try_wait_sleep(bar, parity, POLL_NS);
}
// A time-out: both CTAs' roles see it at their next wait.
__device__ __forceinline__ void record_error(int *err) {
  const uint32_t a = smem_u32(err);
  for (uint32_t k = 0; k < 2; ++k)
    asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(map_cta(a, k)), "r"(1)
                 : "memory");
}
// Bounded wait that only the limit ends early (copies and MMAs in flight).
__device__ __forceinline__ bool wait_done(uint32_t bar) {
  return mbar_wait_sleep_bounded(bar, 0, WAIT_LIMIT, POLL_NS);
}
// Bounded wait that also gives up early once a role has recorded an error.
__device__ __forceinline__ bool wait_phase(uint32_t bar, uint32_t parity, int *err) {
  for (uint32_t it = 0; it < WAIT_LIMIT; ++it) {
    if (try_wait(bar, parity)) return true;
    if ((it & 63u) == 63u && *reinterpret_cast<volatile int *>(err)) return false;
  }
  record_error(err);
  return false;
}
// The same for a whole warp: every lane waits in mbarrier.try_wait (the
// hardware suspends the warp until the phase completes or a short time limit
// passes) and the lanes agree by a vote, so the warp stays converged for the
// .sync.aligned tensor-memory accesses that follow and waiting warps take no
// issue slots from the MMA warp.  (Lane 0 polling test_wait with the other
// lanes held at a shuffle cost 10 % of the step.)
__device__ __forceinline__ bool wait_phase_warp(uint32_t bar, uint32_t parity, int *err) {
  for (uint32_t it = 0; it < WAIT_LIMIT; ++it) {
    if (__any_sync(0xffffffffu, try_wait(bar, parity))) {
      fence_after_sync();
      return true;
    }
    if ((it & 63u) == 63u &&
        __any_sync(0xffffffffu, *reinterpret_cast<volatile int *>(err) != 0))
      return false;
  }
  if ((threadIdx.x & 31) == 0) record_error(err);
  return false;
}
// After this warp's tensor-memory accesses: one arrival at CTA 0's barrier.
__device__ __forceinline__ void publish(uint32_t mapped) {
  tmem_wait_st();
  fence_before_sync();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) arrive_cluster(mapped);
}
// Both CTAs' D (+)= A[tmem] * B[smem halves]^T, one thread of CTA 0.
__device__ __forceinline__ void mma_pair(uint32_t d, uint32_t a_tmem, uint64_t b, uint32_t id,
                                         bool acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
      "r"(a_tmem), "l"(b), "r"(id), "r"(acc ? 1u : 0u)
      : "memory");
}
// Arrive on this barrier of both CTAs when the MMAs issued so far are done.
__device__ __forceinline__ void commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 "
      "[%0], %1;" ::"r"(bar),
      "h"((uint16_t)3)
      : "memory");
}

// A node of the flattened lattice, walked in steps of two tiles.
struct NodePos {
  long long n;
  int x, y, z, b;
};
struct NodeStep {
  int dx, dy, dz, db;
};
__device__ __forceinline__ NodePos locate(const Grid3 &g, long long n) {
  NodePos p;
  p.n = n;
  long long row = n / g.nx;
  p.x = (int)(n - row * g.nx);
  long long pl = row / g.ny;
  p.y = (int)(row - pl * g.ny);
  p.b = (int)(pl / g.nz);
  p.z = (int)(pl - (long long)p.b * g.nz);
  return p;
}
__device__ __forceinline__ void advance(NodePos &p, const Grid3 &g, const NodeStep &d) {
  p.n += 2 * TILE;
  p.x += d.dx;
  int c = p.x >= g.nx;
  p.x -= c ? g.nx : 0;
  p.y += d.dy + c;
  c = p.y >= g.ny;
  p.y -= c ? g.ny : 0;
  p.z += d.dz + c;
  c = p.z >= g.nz;
  p.z -= c ? g.nz : 0;
  p.b += d.db + c;
}

__device__ __forceinline__ void pull19(const float *__restrict__ in, const Grid3 &g,
                                       const NodePos &p, long long nodes, float d[Q]) {
#pragma unroll
  for (int i = 0; i < Q; ++i) d[i] = 0.f;
  if (p.n >= nodes) return;
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

// 16 accumulator columns -> LeakyReLU -> 8 columns of bf16 pairs.  The two
// products 0.01 v of a pair in one packed multiply (round to nearest per lane,
// as the scalar form), then max.
__device__ __forceinline__ void activate16(const uint32_t (&v)[16], uint32_t dst) {
  uint32_t p[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const float a0 = __uint_as_float(v[2 * e]), a1 = __uint_as_float(v[2 * e + 1]);
    const float2 s = __fmul2_rn(make_float2(a0, a1), make_float2(LEAKY, LEAKY));
    p[e] = pack_bf16x2(fmaxf(a0, s.x), fmaxf(a1, s.y));
  }
  tmem_st8(dst, p);
}
// K steps k0 .. k0 + steps - 1 (3 to 5) of a layer's accumulator (from tensor-
// memory column acc on) -> activations at the columns `table` gives.  All
// loads are issued before one wait, so in-place stores follow the loads of the
// columns they replace.  The padding needs no special case: the row after a
// layer's last unit in the prepared weights has its bias 1 and all else 0, so
// its accumulator is the constant input of the next layer, and the rows after
// it are 0.
// One body serves all layers and both warpgroups: a drain compiled for each
// part made the kernel 100 KB long, and most SMs then waited for instructions
// (13.6 k cycles per tile against 9.4 k on the few that did not).
__device__ __forceinline__ void drain(uint32_t tm_row, uint32_t acc, const ColTable &table, int k0,
                                      int steps) {
  uint32_t v[5][16];
  const uint32_t src = tm_row + acc + 16 * k0;
#pragma unroll
  for (int s = 0; s < 3; ++s) tmem_ld16(src + 16 * s, v[s]);
  if (steps > 3) tmem_ld16(src + 48, v[3]);
  if (steps > 4) tmem_ld16(src + 64, v[4]);
  tmem_wait_ld();
#pragma unroll
  for (int s = 0; s < 5; ++s)
    if (s < 3 || steps > s) activate16(v[s], tm_row + table(k0 + s));
}

// x = (f - feq)/rho of this thread's node -> its row of the layer-1 operand
// (19 inputs, the constant-1 bias column, zeros) in tensor memory.
__device__ __forceinline__ void write_x(const float d[Q], bool active, uint32_t tm_row) {
  const Moments m = node_moments(d);
  float deq[Q];
  shifted_feq(m, deq);
  const float inv_rho = 1.0f / m.rho;
  float xi[32];
#pragma unroll
  for (int i = 0; i < 32; ++i)
    xi[i] = i < Q ? (active ? (d[i] - deq[i]) * inv_rho : 0.f) : (i == Q ? 1.0f : 0.0f);
  uint32_t p[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) p[e] = pack_bf16x2(xi[2 * e], xi[2 * e + 1]);
  tmem_st16(tm_row + TM_X, p);
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
    k3_step_mlp_tc(const float *__restrict__ in, float *__restrict__ out, Grid3 g, Collide3 cp,
                   const unsigned char *__restrict__ gw, int *flag, int *timeout_flag) {
  extern __shared__ unsigned char smem_raw[];
  Smem &S = *reinterpret_cast<Smem *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                      ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_rank();
  int *err = &S.err;

  // ---- prologue: barriers, this CTA's half of the weights, tensor memory
  if (tid == 0) {
    mbar_init(smem_u32(&S.bx), 8);
    mbar_init(smem_u32(&S.bo), 8);
    for (unsigned long long *b : {&S.b1lo, &S.b1hi, &S.b2lo, &S.b2hi, &S.b3})
      mbar_init(smem_u32(b), 16);
    for (unsigned long long *b : {&S.c1a, &S.c1b, &S.c2a, &S.c2b, &S.c3, &S.c4, &S.wload, &S.drain[0],
                                  &S.drain[1], &S.drain[2]})
      mbar_init(smem_u32(b), 1);
    S.err = 0;
    fence_mbarrier_init();
    fence_proxy_async();
    const uint32_t bar = smem_u32(&S.wload);
    mbar_arrive_expect_tx(bar, G_BYTES);
    const unsigned char *src = gw + (size_t)rank * G_BYTES;
    for (int at = 0; at < G_BYTES; at += 16384) {
      const uint32_t n = G_BYTES - at < 16384 ? G_BYTES - at : 16384;
      bulk_g2s(smem_u32(S.w) + at, src + at, n, bar);
    }
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                     smem_u32(&S.taddr))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  fence_before_sync();
  __syncthreads();
  cluster_sync();  // both CTAs run, and their error words are set up
  // the weights have landed (bounded; every thread polls, so that all see the copy);
  // if a CTA's have not, neither CTA starts its roles
  if (!wait_done(smem_u32(&S.wload))) record_error(err);
  cluster_sync();
  fence_after_sync();
  const uint32_t tmem = S.taddr;
  // the prologue reads only the prepared weights: launched as a programmatic
  // dependent of the previous step, it waits for that step here
  griddep_wait();
  griddep_launch_dependents();

  // ---- this cluster's contiguous range of tile pairs
  const long long nodes = (long long)g.nx * g.ny * g.nz * g.batch;
  const long long pairs = (nodes + 2 * TILE - 1) / (2 * TILE);
  const int clusters = gridDim.x / 2, cid = blockIdx.x / 2;
  const long long per = pairs / clusters, extra = pairs % clusters;
  const long long p_begin = cid * per + (cid < extra ? cid : extra);
  const int count = (int)(per + (cid < extra ? 1 : 0));
  const bool ok0 = *reinterpret_cast<volatile int *>(err) == 0;

  if (warp >= MMA_WARP) {
    // ---------------- MMA issue: L1 and L2, L3, L4 by a thread each.  (A
    // thread that has committed stalls at its next memory access until its
    // MMAs have completed, so one thread for all would start every layer that
    // much late.)
    if (rank == 0 && lane == 0 && ok0) {
      const uint32_t sw = smem_u32(S.w);
      constexpr uint32_t ID_LO = idesc_bf16_f32(256, NLO), ID_HI = idesc_bf16_f32(256, NHI),
                         ID_3 = idesc_bf16_f32(256, N3), ID_4 = idesc_bf16_f32(256, N4);
      const uint32_t P = tmem + TM_P;
      uint32_t par = 0;  // parity of tile t's events
      if (warp == MMA_WARP) {
        const uint32_t w1lo = sw + G_W1, w1hi = w1lo + R_LO * KX * 2;
        const uint32_t w2lo = sw + G_W2, w2hi = w2lo + R_LO * KH * 2;
        for (int t = 0; t < count; ++t, par ^= 1) {
          // L1: its accumulator replaces the previous tile's h2, so that tile's
          // L3 has to be complete
          if (!(wait_phase(smem_u32(&S.bx), par, err) &&
                (t == 0 || wait_phase(smem_u32(&S.c3), par ^ 1, err))))
            break;
          fence_after_sync();
#pragma unroll
          for (int s = 0; s < KX / 16; ++s)
            mma_pair(P, tmem + TM_X + 8 * s, smem_desc(w1lo + 256 * s, 128, 16 * KX), ID_LO, s > 0);
          commit_pair(smem_u32(&S.c1a));
#pragma unroll
          for (int s = 0; s < KX / 16; ++s)
            mma_pair(P + NLO, tmem + TM_X + 8 * s, smem_desc(w1hi + 256 * s, 128, 16 * KX), ID_HI,
                     s > 0);
          commit_pair(smem_u32(&S.c1b));
          // L2, first pass: the lower half of h1 is ready before the upper one
          if (!wait_phase(smem_u32(&S.b1lo), par, err)) break;
          fence_after_sync();
#pragma unroll
          for (int s = 0; s < NLO / 16; ++s)
            mma_pair(P, tmem + col_h1()(s), smem_desc(w2lo + 256 * s, 128, 16 * KH), ID_LO, s > 0);
          if (!wait_phase(smem_u32(&S.b1hi), par, err)) break;
          fence_after_sync();
#pragma unroll
          for (int s = NLO / 16; s < KH / 16; ++s)
            mma_pair(P, tmem + col_h1()(s), smem_desc(w2lo + 256 * s, 128, 16 * KH), ID_LO, true);
          commit_pair(smem_u32(&S.c2a));
          // second pass
#pragma unroll
          for (int s = 0; s < KH / 16; ++s)
            mma_pair(P + NLO, tmem + col_h1()(s), smem_desc(w2hi + 256 * s, 128, 16 * KH), ID_HI,
                     s > 0);
          commit_pair(smem_u32(&S.c2b));
        }
      } else if (warp == MMA_WARP + 1) {
        // L3: its accumulator replaces h1, so L2 has to be complete
        const uint32_t w3 = sw + G_W3, D3 = tmem + TM_A;
        for (int t = 0; t < count; ++t, par ^= 1) {
          if (!(wait_phase(smem_u32(&S.c2b), par, err) && wait_phase(smem_u32(&S.b2lo), par, err)))
            break;
          fence_after_sync();
#pragma unroll
          for (int s = 0; s < NLO / 16; ++s)
            mma_pair(D3, tmem + col_h2()(s), smem_desc(w3 + 256 * s, 128, 16 * KH), ID_3, s > 0);
          if (!wait_phase(smem_u32(&S.b2hi), par, err)) break;
          fence_after_sync();
#pragma unroll
          for (int s = NLO / 16; s < KH / 16; ++s)
            mma_pair(D3, tmem + col_h2()(s), smem_desc(w3 + 256 * s, 128, 16 * KH), ID_3, true);
          commit_pair(smem_u32(&S.c3));
        }
      } else {
        // L4, once the previous tile's output has been read
        const uint32_t w4 = sw + G_W4;
        for (int t = 0; t < count; ++t, par ^= 1) {
          if (!(wait_phase(smem_u32(&S.b3), par, err) &&
                (t == 0 || wait_phase(smem_u32(&S.bo), par ^ 1, err))))
            break;
          fence_after_sync();
#pragma unroll
          for (int s = 0; s < K4 / 16; ++s)
            mma_pair(tmem + TM_OUT, tmem + col_h3()(s), smem_desc(w4 + 256 * s, 128, 16 * K4), ID_4,
                     s > 0);
          commit_pair(smem_u32(&S.c4));
        }
      }
      // both CTAs wait for this at their end
      commit_pair(smem_u32(&S.drain[warp - MMA_WARP]));
    }
    __syncwarp();
  } else if (warp >= NODE_WARP) {
    // ---------------- node work
    const int r = tid - 32 * NODE_WARP;
    const uint32_t tm_row = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    const uint32_t m_x = map_cta(smem_u32(&S.bx), 0), m_o = map_cta(smem_u32(&S.bo), 0);
    const uint32_t c1 = smem_u32(&S.c1b), c4 = smem_u32(&S.c4);
    const size_t vol = g.volume();
    NodeStep st;
    {
      int q = 2 * TILE / g.nx;
      st.dx = 2 * TILE % g.nx;
      st.dy = q % g.ny;
      q /= g.ny;
      st.dz = q % g.nz;
      st.db = q / g.nz;
    }
    // Iteration t loads tile t + 2, writes the layer-1 operand of tile t + 1 and
    // finishes tile t (one body for all, for the instruction cache).
    NodePos P{}, N{}, F = locate(g, p_begin * 2 * TILE + rank * TILE + r);
    float d[Q], dn[Q], df[Q];  // populations of tiles t, t + 1, t + 2
#pragma unroll
    for (int i = 0; i < Q; ++i) d[i] = dn[i] = df[i] = 0.f;
#pragma unroll 1
    for (int t = -2; t < count && ok0; ++t) {
      const uint32_t par = t & 1;
      if (t + 2 < count) pull19(in, g, F, nodes, df);
      if (t >= -1 && t + 1 < count) {
        if (t >= 0 && !wait_phase_warp(c1, par, err)) break;  // L1 has read x
        write_x(dn, N.n < nodes, tm_row);
        publish(m_x);
      }
      if (t >= 0) {
        const bool active = P.n < nodes;
        const Moments m = node_moments(d);
        {
          const unsigned mask = __ballot_sync(0xffffffffu, active && is_unstable(m));
          if (mask && lane == (__ffs(mask) - 1) && *reinterpret_cast<volatile int *>(flag) == 0)
            atomicOr(flag, 1);
        }
        float deq[Q];
        shifted_feq(m, deq);
        if (!wait_phase_warp(c4, par, err)) break;
        uint32_t v0[16], v1[16];
        tmem_ld16(tm_row + TM_OUT, v0);
        tmem_ld16(tm_row + TM_OUT + 16, v1);
        tmem_wait_ld();
        publish(m_o);
        float o[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) o[i] = __uint_as_float(i < 16 ? v0[i] : v1[i - 16]);
        project(o);
        if (active) {
          const float rw = m.rho * cp.omega;
#pragma unroll
          for (int i = 0; i < Q; ++i) d[i] = fmaf(cp.omega, deq[i] - d[i], d[i]) + rw * o[i];
          const float Fx = cp.fx_y ? __ldg(cp.fx_y + P.y) : 0.f;
          const float Fy = cp.fy_z ? __ldg(cp.fy_z + P.z) : 0.f;
          const float Fz = cp.fz_x ? __ldg(cp.fz_x + P.x) : 0.f;
          add_edm_force(m, Fx, Fy, Fz, d);
          float *ob = out + (size_t)P.b * Q * vol + ((size_t)P.z * g.ny + P.y) * g.nx + P.x;
#pragma unroll
          for (int i = 0; i < Q; ++i) ob[(size_t)i * vol] = d[i];
        }
      }
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        d[i] = dn[i];
        dn[i] = df[i];
      }
      P = N;
      N = F;
      advance(F, g, st);
    }
  } else if (ok0) {
    // ---------------- epilogues: WG0 the first, WG1 the second columns of each part
    const int wg = warp >> 2;
    const uint32_t tm_row = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    const uint32_t m_1lo = map_cta(smem_u32(&S.b1lo), 0), m_1hi = map_cta(smem_u32(&S.b1hi), 0),
                   m_2lo = map_cta(smem_u32(&S.b2lo), 0), m_2hi = map_cta(smem_u32(&S.b2hi), 0),
                   m_3 = map_cta(smem_u32(&S.b3), 0);
    const uint32_t c1a = smem_u32(&S.c1a), c1b = smem_u32(&S.c1b), c2a = smem_u32(&S.c2a),
                   c2b = smem_u32(&S.c2b), c3 = smem_u32(&S.c3), c4 = smem_u32(&S.c4);
    uint32_t par = 0;
    bool ok = true;
    for (int t = 0; t < count && ok; ++t, par ^= 1) {
      // parts: lower and upper half of h1, of h2, then h3
#pragma unroll 1
      for (int e = 0; e < 5; ++e) {
        // (the upper half of h1 takes columns that h3 of the previous tile held)
        const uint32_t bar = e == 0 ? c1a : e == 1 ? c1b : e == 2 ? c2a : e == 3 ? c2b : c3;
        if (!wait_phase_warp(bar, par, err) ||
            (e == 1 && t > 0 && !wait_phase_warp(c4, par ^ 1, err))) {
          ok = false;
          break;
        }
        const int k0 = (e == 4 ? 4 : 5) * wg + (e & 1 ? 10 : 0);
        const int steps = wg == 0 ? (e == 4 ? 4 : 5) : (e == 4 ? 3 : e & 1 ? 4 : 5);
        const ColTable table = e < 2 ? col_h1() : e < 4 ? col_h2() : col_h3();
        drain(tm_row, e < 4 ? TM_P : TM_A, table, k0, steps);
        publish(e == 0 ? m_1lo : e == 1 ? m_1hi : e == 2 ? m_2lo : e == 3 ? m_2hi : m_3);
      }
    }
  }

  // ---- teardown: every role of both CTAs has left its loop (normally or on an error).
  // The issuers' last commits arrive in both CTAs, and each CTA waits for its own
  // copies of them: no MMA is outstanding when the tensor memory is freed, and no
  // arrival is on its way to a CTA that has left.  (A cluster barrier orders what
  // threads did, not the arrivals of a commit.)
  if (tid < 3 && ok0 && !wait_done(smem_u32(&S.drain[tid]))) record_error(err);
  // (a copy that was late is waited for once more, so that none is in flight at the exit)
  if (tid == 0) wait_done(smem_u32(&S.wload));
  __syncwarp();
  fence_before_sync();
  cluster_sync();
  fence_after_sync();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  if (tid == 0 && S.err) atomicOr(timeout_flag, 1);
}

// FP32 packed weights -> BF16 operand tiles in the canonical K-major layout,
// biases in the constant-1 K column; one block of G_BYTES per CTA of a pair.
__global__ void k3_prepare_weights(Mlp3 w, unsigned char *__restrict__ gw) {
  const int total = NH * KX + N4 * K4 + N3 * KH + NH * KH;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    float v = 0.f;
    int rank;
    size_t off;
    // rows of a hidden matrix: pass 0 | pass 1, each split between the CTAs
    auto place_hidden = [&](int n, int k, int K, int base) {
      const int hi = n >= NLO, m = hi ? n - NLO : n, half = hi ? R_HI : R_LO;
      rank = m >= half;
      off = base + (hi ? R_LO * K * 2 : 0) + canon_offset(m - rank * half, k, K);
    };
    // the row after a hidden layer's last unit yields the constant 1
    auto one = [](bool here) { return here ? 1.f : 0.f; };
    if (e < NH * KX) {  // W1: rows n < 300, K 19 inputs, bias at k = 19
      const int n = e / KX, k = e % KX;
      v = n < H1 ? (k < Q ? w.w1[n * Q + k] : (k == Q ? w.b1[n] : 0.f)) : one(n == H1 && k == Q);
      place_hidden(n, k, KX, G_W1);
    } else if (e < NH * KX + N4 * K4) {  // W4: rows n < 19, K 100, bias at k = 100
      const int f = e - NH * KX, n = f / K4, k = f % K4;
      if (n < Q) v = k < H3 ? w.w4[n * H3 + k] : (k == H3 ? w.b4[n] : 0.f);
      rank = n >= N4 / 2;
      off = G_W4 + canon_offset(n - rank * (N4 / 2), k, K4);
    } else if (e < NH * KX + N4 * K4 + N3 * KH) {  // W3: rows n < 100, K 300, bias at 300
      const int f = e - NH * KX - N4 * K4, n = f / KH, k = f % KH;
      v = n < H3 ? (k < H2 ? w.w3[n * H2 + k] : (k == H2 ? w.b3[n] : 0.f)) : one(n == H3 && k == H2);
      rank = n >= N3 / 2;
      off = G_W3 + canon_offset(n - rank * (N3 / 2), k, KH);
    } else {  // W2: rows n < 300, K 300, bias at 300
      const int f = e - NH * KX - N4 * K4 - N3 * KH, n = f / KH, k = f % KH;
      v = n < H2 ? (k < H1 ? w.w2[n * H1 + k] : (k == H1 ? w.b2[n] : 0.f)) : one(n == H2 && k == H1);
      place_hidden(n, k, KH, G_W2);
    }
    *reinterpret_cast<__nv_bfloat16 *>(gw + (size_t)rank * G_BYTES + off) = __float2bfloat16_rn(v);
  }
}

}  // namespace

size_t mlp_tc_weight_bytes() { return 2 * (size_t)G_BYTES; }

cudaError_t launch_prepare_weights_tc(const Mlp3 &w, void *gw, cudaStream_t s) {
  k3_prepare_weights<<<256, 256, 0, s>>>(w, static_cast<unsigned char *>(gw));
  return cudaGetLastError();
}

cudaError_t launch_step_mlp_tc(const Grid3 &g, const float *in, float *out, const Collide3 &c,
                               const void *gw, int sms, int *flag, int *timeout_flag, bool chain,
                               cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(k3_step_mlp_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const long long pairs = ((long long)g.nodes() + 2 * TILE - 1) / (2 * TILE);
  long long clusters = sms / 2;
  if (clusters < 1) return cudaErrorInvalidConfiguration;
  if (pairs < clusters) clusters = pairs;
  if ((pairs + clusters - 1) / clusters > 0x7fffffffLL) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * clusters));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = SMEM_BYTES;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chain ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k3_step_mlp_tc, in, out, g, c,
                            static_cast<const unsigned char *>(gw), flag, timeout_flag);
}

}  // namespace d3
}  // namespace lbm
