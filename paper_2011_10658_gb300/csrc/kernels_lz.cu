// One Lanczos step (three-term residual, full reorthogonalisation, norm) as a
// single persistent launch.
//
// The step is two passes over the Krylov basis (V^T w', then w' - V c) with a
// few scalars in between.  The grid is resident as a whole (cooperative
// launch): every thread owns the same rows in every phase, so only scalars
// cross blocks, through partial sums between grid barriers.
//
// A dot phase takes eight basis columns at a time, each thread summing its
// rows in registers; a warp then exchanges halves of the eight sums (four,
// two, one), which costs nine FP64 additions where eight separate reductions
// cost forty: on GB300's FP64 pipes the additions of a reduction cost as much
// as the products.
//
// Bound by HBM and the FP64 additions at bottom nodes (n = 1.7 M: 222 us a step
// on average over 1-56 vectors, 365 with 56; eleven launches took 560 with 48),
// by the latency of its barriers and loads at upper nodes (n = 5104: 17 us; 25-55
// in the long form).  Whole updates, GB300: bottom node of 4x4x4 chi=64 48.0 ->
// 26 ms, layer 3 at chi=32 14.0 -> 5.9 ms, with the faster products.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "ffloat.cuh"
#include "kernels.cuh"

namespace qed {

namespace {

constexpr int LZ_THREADS = 256;
constexpr int LZ_WARPS = LZ_THREADS / 32;
constexpr int LZ_COLS = 8;                       // basis columns of a dot sweep
constexpr int LZ_MAX_K = 128;
constexpr int LZ_ROW_BLOCKS = kLzRowBlocks;      // row blocks of a sum
constexpr int LZ_ALPHA_BLOCKS = 304;             // of alpha
constexpr int LZ_LONG_BLOCKS = 4;                // most resident blocks per SM of the long form
constexpr int LZ_SHORT = 64;                     // row blocks of the short form
constexpr int LZ_DEVICES = 64;
constexpr int LZ_DIRECT = 64;                    // grids up to this size: every block adds all partial sums itself
constexpr long long kLzPolls = 1LL << 22;        // default bound of a grid barrier's wait (seconds)

__device__ __forceinline__ unsigned lz_load(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Barrier of the whole grid; round counts them.  A wait that runs out sets
// *err and goes on: every access stays in bounds whatever the sums hold, and the
// host rejects the run.
__device__ __forceinline__ void grid_sync(const LzStep& p, unsigned& round) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(p.bar, 1u);
    const unsigned want = ++round * gridDim.x;
    bool ok = false;
    for (long long it = 0; it < p.polls && !ok; ++it) ok = lz_load(p.bar) >= want;
    if (!ok) atomicExch(p.err, 1);
  } else {
    ++round;
  }
  __syncthreads();
}

// ---- sums in a fixed order
// A sum over the rows does not depend on the grid: row block b of LZ_ROW_BLOCKS
// (LZ_ALPHA_BLOCKS for alpha) holds rows 256 b + t, then 256 LZ_ROW_BLOCKS rows
// further on, one chain per t; a warp's 32 chains are added in halves (16, 8,
// 4, 2, 1), its eight warps either one after another (columns of a dot phase)
// or in halves again (single sums), and the row blocks as if they were rows.
// A node update in reduced precision rounds its vectors to FP32 in every
// product, so one changed last place in a coefficient ends as a difference of
// 1e-4 in the update; with this order the launch geometry is free.
__host__ __device__ __forceinline__ int lz_row_blocks(long long n, int most) {
  return (int)(n < (long long)most * LZ_THREADS ? (n + LZ_THREADS - 1) / LZ_THREADS : most);
}

__device__ __forceinline__ double lz_halves8(const double* s) {
  return ((s[0] + s[4]) + (s[2] + s[6])) + ((s[1] + s[5]) + (s[3] + s[7]));
}

__device__ __forceinline__ double lz_warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Eight warp sums at once: lane l ends with the sum of v[(l >> 2) & 7] with its
// bits reversed as 4 (lane bit 4), 2 (bit 3), 1 (bit 2): lz_slot.
__device__ __forceinline__ double lz_warp_sum8(double* v, int lane) {
#pragma unroll
  for (int h = LZ_COLS / 2, m = 16; h >= 1; h >>= 1, m >>= 1)
#pragma unroll
    for (int t = 0; t < h; ++t) {
      const bool up = (lane & m) != 0;
      const double keep = up ? v[t + h] : v[t];
      const double give = up ? v[t] : v[t + h];
      v[t] = keep + __shfl_xor_sync(0xffffffffu, give, m);
    }
  double r = v[0];
  r += __shfl_xor_sync(0xffffffffu, r, 2);
  r += __shfl_xor_sync(0xffffffffu, r, 1);
  return r;
}
__device__ __forceinline__ int lz_slot(int lane) { return ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1); }

// Sum over the block, valid in every thread.
__device__ __forceinline__ double lz_block_sum(double v, double* red) {
  v = lz_warp_sum(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  const double r = lz_halves8(red);
  __syncthreads();
  return r;
}

// Sum of the values of `count` row blocks by one warp, valid in every lane.
__device__ __forceinline__ double lz_total(const double* part, int count, int lane) {
  double v[LZ_COLS];
#pragma unroll
  for (int w = 0; w < LZ_COLS; ++w) v[w] = 0.0;
  for (int base = 0; base < count; base += LZ_THREADS)
#pragma unroll
    for (int w = 0; w < LZ_COLS; ++w) {
      const int i = base + 32 * w + lane;
      if (i < count) v[w] += __ldcg(part + i);
    }
  double r = lz_warp_sum8(v, lane);
  r += __shfl_xor_sync(0xffffffffu, r, 16);
  r += __shfl_xor_sync(0xffffffffu, r, 8);
  r += __shfl_xor_sync(0xffffffffu, r, 4);
  return r;
}

// The same, valid in every thread.
__device__ __forceinline__ double lz_grid_sum(const double* part, int count, double* red) {
  if (threadIdx.x < 32) {
    const double r = lz_total(part, count, threadIdx.x);
    if (threadIdx.x == 0) red[0] = r;
  }
  __syncthreads();
  const double r = red[0];
  __syncthreads();
  return r;
}

// One thread's products V_col . row for the columns g .. g + 7 (col = k: row .
// row), for its rows of a row block; then summed over the warp.
template <typename A, typename Row>
__device__ __forceinline__ double lz_dot8(const LzStep& p, int g, long long i0, long long step, int lane, Row row) {
  A acc[LZ_COLS];
#pragma unroll
  for (int t = 0; t < LZ_COLS; ++t) acc[t] = A(0);
  const int cols = min(LZ_COLS, p.k - g);   // basis columns among them
  if (cols == LZ_COLS) {
#pragma unroll 1
    for (long long i = i0; i < p.n; i += step) {
      const double* q = p.V + (long long)g * p.ldq + i;
      double v[LZ_COLS];
#pragma unroll
      for (int t = 0; t < LZ_COLS; ++t, q += p.ldq) v[t] = __ldg(q);
      const A ya = raw_t<A>(row(i));
#pragma unroll
      for (int t = 0; t < LZ_COLS; ++t) acc[t] = kc_fma(raw_t<A>(v[t]), ya, acc[t]);
    }
  } else {
#pragma unroll 1
    for (long long i = i0; i < p.n; i += step) {
      const double* q = p.V + (long long)g * p.ldq + i;
      double v[LZ_COLS];
#pragma unroll
      for (int t = 0; t < LZ_COLS; ++t, q += p.ldq) v[t] = t < cols ? __ldg(q) : 0.0;
      const A ya = raw_t<A>(row(i));
#pragma unroll
      for (int t = 0; t < LZ_COLS; ++t) {
        if (t < cols) acc[t] = kc_fma(raw_t<A>(v[t]), ya, acc[t]);
        else if (t == cols) acc[t] = kc_fma(ya, ya, acc[t]);
      }
    }
  }
  double s[LZ_COLS];
#pragma unroll
  for (int t = 0; t < LZ_COLS; ++t) s[t] = to_d<A>(acc[t]);
  return lz_warp_sum8(s, lane);
}

// y_i - sum_j c_j V_j[i], columns in order.
template <typename A>
__device__ __forceinline__ A lz_minus(const LzStep& p, const A* cs, double y, long long i) {
  A v = raw_t<A>(y);
  const double* q = p.V + i;
  int j = 0;
  for (; j + LZ_COLS <= p.k; j += LZ_COLS) {
    double x[LZ_COLS];
#pragma unroll
    for (int t = 0; t < LZ_COLS; ++t, q += p.ldq) x[t] = __ldg(q);
#pragma unroll
    for (int t = 0; t < LZ_COLS; ++t) v = kc_fma(cs[j + t], raw_t<A>(x[t]), v);
  }
  for (; j < p.k; ++j, q += p.ldq) v = kc_fma(cs[j], raw_t<A>(__ldg(q)), v);
  return v;
}

// partial[col * blocks + b] = row block b's V_col . y for col < k, and y . y
// for col = k.
template <typename A>
__device__ __forceinline__ void lz_dots(const LzStep& p, int blocks, double (*sh)[LZ_MAX_K + LZ_COLS]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long step = (long long)LZ_ROW_BLOCKS * LZ_THREADS;
  for (int b = blockIdx.x; b < blocks; b += gridDim.x) {
    const long long i0 = (long long)b * LZ_THREADS + threadIdx.x;
    for (int g = 0; g <= p.k; g += LZ_COLS) {
      const double r = lz_dot8<A>(p, g, i0, step, lane, [&](long long i) { return p.y[i]; });
      if ((lane & 3) == 0) sh[warp][g + lz_slot(lane)] = r;
    }
    __syncthreads();
    if ((int)threadIdx.x <= p.k) {
      double v = 0.0;
#pragma unroll
      for (int u = 0; u < LZ_WARPS; ++u) v += sh[u][threadIdx.x];
      __stcg(p.partial + (long long)threadIdx.x * blocks + b, v);
    }
    __syncthreads();
  }
}

// c[col] = sum over the row blocks of partial[col], col < ncol, in every
// block's shared memory.  Large grids: one warp of the grid a column first.
__device__ __forceinline__ void lz_columns(const LzStep& p, int ncol, int blocks, double* coef, double* c,
                                           unsigned& round) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool direct = (int)gridDim.x <= LZ_DIRECT;
  const int first = direct ? warp : (int)blockIdx.x + (int)gridDim.x * warp;
  const int step = direct ? LZ_WARPS : (int)gridDim.x * LZ_WARPS;
  for (int col = first; col < ncol; col += step) {
    const double v = lz_total(p.partial + (long long)col * blocks, blocks, lane);
    if (lane == 0) {
      if (direct) c[col] = v;
      else __stcg(coef + col, v);
    }
  }
  if (!direct) {
    grid_sync(p, round);
    for (int col = threadIdx.x; col < ncol; col += LZ_THREADS) c[col] = __ldcg(coef + col);
  }
  __syncthreads();
}

// y -= V c; part[b] = row block b's part of |y|^2.
template <typename A>
__device__ __forceinline__ void lz_update(const LzStep& p, int blocks, const double* c, A* cs, double* part,
                                          double* red) {
  for (int j = threadIdx.x; j < p.k; j += LZ_THREADS) cs[j] = raw_t<A>(-c[j]);
  __syncthreads();
  const long long step = (long long)LZ_ROW_BLOCKS * LZ_THREADS;
  for (int b = blockIdx.x; b < blocks; b += gridDim.x) {
    A nrm = A(0);
#pragma unroll 2
    for (long long i = (long long)b * LZ_THREADS + threadIdx.x; i < p.n; i += step) {
      const A v = lz_minus<A>(p, cs, p.y[i], i);
      p.y[i] = to_d<A>(v);
      nrm = kc_fma(v, v, nrm);
    }
    const double s = lz_block_sum(to_d<A>(nrm), red);
    if (threadIdx.x == 0) __stcg(part + b, s);
  }
}

// A wait ran out, in this launch or before it.
__device__ __forceinline__ bool lz_failed(const LzStep& p) { return lz_load((const unsigned*)p.err) != 0u; }

// The last block to leave zeroes the counters for the next launch.
__device__ __forceinline__ void lz_leave(const LzStep& p, double alpha, double nrm2) {
  if (threadIdx.x == 0) {
    if (blockIdx.x == 0) {
      const bool failed = lz_failed(p);
      *p.alpha_j = failed ? 0.0 : alpha;
      *p.beta_j = failed ? 0.0 : sqrt(fmax(nrm2, 0.0));
    }
    if (atomicAdd(p.bar + 1, 1u) == gridDim.x - 1) {
      p.bar[0] = 0u;
      p.bar[1] = 0u;
    }
  }
}

// ---- short vectors: the basis columns are shared out as well
// Block (rb, cg) of row_blocks x column_groups: row block rb, column sweeps cg,
// cg + column_groups, ..  A short vector leaves a thread one row, so the time
// is the number of trips to L2 one after another; here a dot phase is one sweep
// per block, and the warps of an update are spread over all blocks.
// part[rb * (k + 1) + col]; `row` gives w' (or y) of a row.
template <typename A, typename Row>
__device__ __forceinline__ void lz_short_dots(const LzStep& p, int rb, int cg, int column_groups,
                                              double (*sh)[LZ_MAX_K + LZ_COLS], Row row) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int g = cg * LZ_COLS; g <= p.k; g += column_groups * LZ_COLS) {
    const double r = lz_dot8<A>(p, g, (long long)rb * LZ_THREADS + threadIdx.x, p.n, lane, row);
    if ((lane & 3) == 0) sh[warp][lz_slot(lane)] = r;
    __syncthreads();
    if (threadIdx.x < LZ_COLS && g + (int)threadIdx.x <= p.k) {
      double v = 0.0;
#pragma unroll
      for (int u = 0; u < LZ_WARPS; ++u) v += sh[u][threadIdx.x];
      __stcg(p.partial + (long long)rb * (p.k + 1) + g + threadIdx.x, v);
    }
    __syncthreads();
  }
}

// c[col] = sum over the (at most 64) row blocks, in every block, a warp eight
// columns at a time.
__device__ __forceinline__ void lz_short_columns(const LzStep& p, int ncol, int row_blocks, double* c) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int g = warp * LZ_COLS; g < ncol; g += LZ_WARPS * LZ_COLS) {
    double v[2][LZ_COLS];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int t = 0; t < LZ_COLS; ++t)
        v[h][t] = lane + 32 * h < row_blocks && g + t < ncol
                      ? __ldcg(p.partial + (long long)(lane + 32 * h) * (p.k + 1) + g + t)
                      : 0.0;
    double r = lz_warp_sum8(v[0], lane);
    if (row_blocks > 32) r += lz_warp_sum8(v[1], lane);
    if ((lane & 3) == 0 && g + lz_slot(lane) < ncol) c[g + lz_slot(lane)] = r;
  }
  __syncthreads();
}

// y = row - V c, a lane a row; part[u] = |y|^2 over rows 32 u .. 32 u + 31.
template <typename A, typename Row>
__device__ __forceinline__ void lz_short_update(const LzStep& p, int row_blocks, const double* c, A* cs, double* part,
                                                Row row) {
  for (int j = threadIdx.x; j < p.k; j += LZ_THREADS) cs[j] = raw_t<A>(-c[j]);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int u = (int)blockIdx.x + (int)gridDim.x * (threadIdx.x >> 5); u < row_blocks * LZ_WARPS;
       u += (int)gridDim.x * LZ_WARPS) {
    const long long i = 32LL * u + lane;
    A nrm = A(0);
    if (i < p.n) {
      const A v = lz_minus<A>(p, cs, row(i), i);
      p.y[i] = to_d<A>(v);
      nrm = kc_fma(v, v, nrm);
    }
    const double s = lz_warp_sum(to_d<A>(nrm));
    if (lane == 0) __stcg(part + u, s);
  }
}

// Sum of the warp sums of at most 64 row blocks, valid in every thread.
__device__ __forceinline__ double lz_short_sum(const double* part, int row_blocks, double* red) {
  if (threadIdx.x < 32) {
    double r = 0.0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int b = threadIdx.x + 32 * h;
      double s[LZ_WARPS];
#pragma unroll
      for (int u = 0; u < LZ_WARPS; ++u) s[u] = b < row_blocks ? __ldcg(part + b * LZ_WARPS + u) : 0.0;
      if (32 * h < row_blocks) r += lz_warp_sum(lz_halves8(s));
    }
    if (threadIdx.x == 0) red[0] = r;
  }
  __syncthreads();
  const double r = red[0];
  __syncthreads();
  return r;
}

template <bool FF>
__global__ void __launch_bounds__(LZ_THREADS, 3) lz_short_kernel(LzStep p, int row_blocks, int column_groups) {
  using A = typename std::conditional<FF, ff, double>::type;
  __shared__ double sh[LZ_WARPS][LZ_MAX_K + LZ_COLS];
  __shared__ double c[LZ_MAX_K + 4];
  __shared__ A cs[LZ_MAX_K];
  double* red = &sh[0][0];
  // one reader per block: another block may set the flag meanwhile
  if (__syncthreads_or(threadIdx.x == 0 && lz_failed(p))) {
    lz_leave(p, 0.0, 0.0);
    return;
  }
  unsigned round = 0;
  const int rb = blockIdx.x % row_blocks, cg = blockIdx.x / row_blocks;
  const double* vj = p.V + (long long)(p.k - 1) * p.ldq;
  const double* vp = vj - p.ldq;
  double* part_a = p.partial + (long long)(LZ_MAX_K + 1) * LZ_ROW_BLOCKS;
  double* part_b = part_a + LZ_ROW_BLOCKS;
  if (cg == 0) {
    const long long i = (long long)rb * LZ_THREADS + threadIdx.x;
    const double a = lz_block_sum(i < p.n ? __ldg(vj + i) * __ldcg(p.y + i) : 0.0, red);
    if (threadIdx.x == 0) __stcg(part_a + rb, a);
  }
  grid_sync(p, round);
  const double alpha = lz_grid_sum(part_a, row_blocks, red);
  const double beta = p.k >= 2 ? *p.beta_prev : 0.0;
  // w' of a row, formed wherever it is needed: y is written in the update only
  auto residual = [&](long long i) {
    double v = fma(-alpha, __ldg(vj + i), __ldcg(p.y + i));
    return p.k >= 2 ? fma(-beta, __ldg(vp + i), v) : v;
  };
  lz_short_dots<A>(p, rb, cg, column_groups, sh, residual);
  grid_sync(p, round);
  lz_short_columns(p, p.k + 1, row_blocks, c);
  const double before = c[p.k];
  lz_short_update<A>(p, row_blocks, c, cs, part_b, residual);
  grid_sync(p, round);
  double nrm2 = lz_short_sum(part_b, row_blocks, red);
  if (nrm2 < p.ratio * before) {
    auto plain = [&](long long i) { return __ldcg(p.y + i); };
    lz_short_dots<A>(p, rb, cg, column_groups, sh, plain);
    grid_sync(p, round);
    lz_short_columns(p, p.k, row_blocks, c);
    lz_short_update<A>(p, row_blocks, c, cs, part_a, plain);
    grid_sync(p, round);
    nrm2 = lz_short_sum(part_a, row_blocks, red);
  }
  const double inv = 1.0 / sqrt(nrm2);
  for (long long i = blockIdx.x * (long long)LZ_THREADS + threadIdx.x; i < p.n; i += (long long)gridDim.x * LZ_THREADS)
    p.v_next[i] = __ldcg(p.y + i) * inv;
  lz_leave(p, alpha, nrm2);
}

template <bool FF>
__global__ void __launch_bounds__(LZ_THREADS, LZ_LONG_BLOCKS) lz_step_kernel(LzStep p) {
  using A = typename std::conditional<FF, ff, double>::type;
  __shared__ double sh[LZ_WARPS][LZ_MAX_K + LZ_COLS];
  __shared__ double c[LZ_MAX_K + 4];
  __shared__ A cs[LZ_MAX_K];
  double* red = &sh[0][0];
  // one reader per block: another block may set the flag meanwhile
  if (__syncthreads_or(threadIdx.x == 0 && lz_failed(p))) {
    lz_leave(p, 0.0, 0.0);
    return;
  }
  unsigned round = 0;
  const int blocks = lz_row_blocks(p.n, LZ_ROW_BLOCKS), blocks_a = lz_row_blocks(p.n, LZ_ALPHA_BLOCKS);
  const double* vj = p.V + (long long)(p.k - 1) * p.ldq;
  const double* vp = vj - p.ldq;
  double* part_a = p.partial + (long long)(LZ_MAX_K + 1) * LZ_ROW_BLOCKS;
  double* part_b = part_a + LZ_ROW_BLOCKS;
  // alpha_j = v_j . y
  for (int b = blockIdx.x; b < blocks_a; b += gridDim.x) {
    double a = 0.0;
#pragma unroll 4
    for (long long i = (long long)b * LZ_THREADS + threadIdx.x; i < p.n; i += (long long)LZ_ALPHA_BLOCKS * LZ_THREADS)
      a = fma(__ldg(vj + i), __ldcg(p.y + i), a);
    a = lz_block_sum(a, red);
    if (threadIdx.x == 0) __stcg(part_a + b, a);
  }
  grid_sync(p, round);
  const double alpha = lz_grid_sum(part_a, blocks_a, red);
  // w' = y - alpha_j v_j - beta_{j-1} v_{j-1}; a thread keeps its rows from here on
  const double beta = p.k >= 2 ? *p.beta_prev : 0.0;
  for (int b = blockIdx.x; b < blocks; b += gridDim.x)
#pragma unroll 2
    for (long long i = (long long)b * LZ_THREADS + threadIdx.x; i < p.n; i += (long long)LZ_ROW_BLOCKS * LZ_THREADS) {
      double v = fma(-alpha, __ldg(vj + i), __ldcg(p.y + i));
      if (p.k >= 2) v = fma(-beta, __ldg(vp + i), v);
      p.y[i] = v;
    }
  lz_dots<A>(p, blocks, sh);
  grid_sync(p, round);
  lz_columns(p, p.k + 1, blocks, p.coef, c, round);
  const double before = c[p.k];
  lz_update<A>(p, blocks, c, cs, part_b, red);
  grid_sync(p, round);
  double nrm2 = lz_grid_sum(part_b, blocks, red);
  if (nrm2 < p.ratio * before) {
    lz_dots<A>(p, blocks, sh);
    grid_sync(p, round);
    lz_columns(p, p.k, blocks, p.coef, c, round);
    lz_update<A>(p, blocks, c, cs, part_a, red);
    grid_sync(p, round);
    nrm2 = lz_grid_sum(part_a, blocks, red);
  }
  const double inv = 1.0 / sqrt(nrm2);
  for (int b = blockIdx.x; b < blocks; b += gridDim.x)
#pragma unroll 2
    for (long long i = (long long)b * LZ_THREADS + threadIdx.x; i < p.n; i += (long long)LZ_ROW_BLOCKS * LZ_THREADS)
      p.v_next[i] = p.y[i] * inv;
  lz_leave(p, alpha, nrm2);
}

}  // namespace

// Vectors of up to 16384 rows: a row per thread in the dots, the column sweeps
// on further blocks.  Longer ones: two row blocks a block up to the resident
// maximum, four blocks an SM, which divides the 1216 of a long vector evenly
// (n = 1.7 M, 1-56 vectors: 222 us a step on average, 272 with three an SM, 316
// with two; n = 100 k in FP64: 77 us, 97 with one row block a block).
int launch_lz_step(const LzStep& p, int ff_arith, cudaStream_t s) {
  if (p.k < 1 || p.k > LZ_MAX_K) return -7;
  int row_blocks = lz_row_blocks(p.n, LZ_ROW_BLOCKS);
  int dev = 0;
  cudaGetDevice(&dev);
  static std::atomic<int> resident[LZ_DEVICES][4];   // blocks a device holds at once, per kernel
  const void* kern = nullptr;
  int cap = 0;
  bool is_short = row_blocks <= LZ_SHORT;
  for (int attempt = 0; attempt < 2; ++attempt) {
    kern = is_short ? (ff_arith ? (const void*)lz_short_kernel<true> : (const void*)lz_short_kernel<false>)
                    : (ff_arith ? (const void*)lz_step_kernel<true> : (const void*)lz_step_kernel<false>);
    std::atomic<int>& known = resident[dev % LZ_DEVICES][(ff_arith ? 1 : 0) + (is_short ? 2 : 0)];
    if (!known || dev >= LZ_DEVICES) {
      int sms = 0, per = 0;
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, LZ_THREADS, 0);
      known = std::max(1, std::min(is_short ? 3 : LZ_LONG_BLOCKS, per) * sms);
    }
    cap = known;
    if (!is_short || row_blocks <= cap) break;
    is_short = false;   // a row block of the short form needs a block of its own
  }
  LzStep arg = p;
  if (arg.polls < 0) arg.polls = kLzPolls;
  int column_groups = std::max(1, std::min(cap / row_blocks, (p.k + LZ_COLS) / LZ_COLS));
  const int blocks = is_short ? row_blocks * column_groups : std::min(cap, (row_blocks + 1) / 2);
  void* args[] = {&arg, &row_blocks, &column_groups};
  if (cudaLaunchCooperativeKernel(kern, dim3(blocks), dim3(LZ_THREADS), args, 0, s) != cudaSuccess) return -3;
  count_launches(1);
  return 0;
}

}  // namespace qed
