// One Lanczos step (three-term residual, full reorthogonalisation, norm) as a
// single persistent launch.
//
// The step is two passes over the Krylov basis (V^T w', then w' - V c) with a
// few scalars in between.  The grid is resident as a whole (cooperative
// launch): every thread owns the same rows in every phase, so only scalars
// cross blocks, through per-block partial sums that are added in block order
// (the result does not depend on scheduling) between grid barriers.
//
// A dot phase takes eight basis columns at a time, each thread summing its
// rows in registers; a warp then exchanges halves of the eight sums (four,
// two, one), which costs nine additions where eight separate reductions cost
// forty -- on GB300's FP64 pipes, and in float-float arithmetic on the FP32
// pipes, the additions of a reduction cost as much as the products.
//
// Bound by HBM at bottom nodes (n = 1.7 M, 48 vectors: 331 us for 1.5 GB with
// the pass over y, 5.2 TB/s per added column; eleven launches took 560), by
// the latency of its barriers and loads at upper nodes.  Whole updates, GB300:
// bottom node of 4x4x4 chi=64 48.0 -> 34.5 ms, layer 3 at chi=32 13.7 -> 9.7
// ms; FP64 sweep of 2x2x2 chi=8 192 -> 129 ms.
#include <algorithm>
#include <type_traits>

#include "ffloat.cuh"
#include "kernels.cuh"

namespace qed {

namespace {

constexpr int LZ_THREADS = 256;
constexpr int LZ_WARPS = LZ_THREADS / 32;
constexpr int LZ_COLS = 8;                       // basis columns of a dot sweep
constexpr int LZ_MAX_K = 128;
constexpr int LZ_DIRECT = 64;                    // grids up to this size: every block adds all partial sums itself
constexpr long long kLzPolls = 1LL << 22;        // bound of a grid barrier's wait (seconds)

// Operands as they come: the sums' own rounding is above what to_t would save.
template <typename A>
__device__ __forceinline__ A lz_in(double v) { return v; }
template <>
__device__ __forceinline__ ff lz_in<ff>(double v) { return d2ff(v); }

template <typename A>
__device__ __forceinline__ A lz_xor(A v, int m);
template <>
__device__ __forceinline__ double lz_xor<double>(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
template <>
__device__ __forceinline__ ff lz_xor<ff>(ff v, int m) {
  return ff(__shfl_xor_sync(0xffffffffu, v.hi, m), __shfl_xor_sync(0xffffffffu, v.lo, m));
}

__device__ __forceinline__ unsigned lz_load(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Barrier of the whole grid; round counts them.  A wait that runs out sets
// *err and goes on (the host then rejects the step).
__device__ __forceinline__ void grid_sync(unsigned* bar, unsigned& round, int* err) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    const unsigned want = ++round * gridDim.x;
    bool ok = false;
    for (long long it = 0; it < kLzPolls && !ok; ++it) ok = lz_load(bar) >= want;
    if (!ok) atomicExch(err, 1);
  } else {
    ++round;
  }
  __syncthreads();
}

// Sum over the block, valid in every thread.
template <typename A>
__device__ __forceinline__ double lz_block_sum(A v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v = v + lz_xor(v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = to_d<A>(v);
  __syncthreads();
  double r = 0.0;
#pragma unroll
  for (int u = 0; u < LZ_WARPS; ++u) r += red[u];
  __syncthreads();
  return r;
}

// Sum of `count` values (one per block), in block order by lanes; valid in
// every thread.
__device__ __forceinline__ double lz_grid_sum(const double* part, int count, double* red) {
  if (threadIdx.x < 32) {
    double v = 0.0;
#pragma unroll 4
    for (int i = threadIdx.x; i < count; i += 32) v += __ldcg(part + i);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) red[0] = v;
  }
  __syncthreads();
  const double r = red[0];
  __syncthreads();
  return r;
}

// part[col * gridDim.x + block] = this block's V_col . y for col < k, and y . y
// for col = k.
template <typename A>
__device__ __forceinline__ void lz_dots(const LzStep& p, double (*sh)[LZ_COLS], long long i0, long long step) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int g = 0; g <= p.k; g += LZ_COLS) {
    A acc[LZ_COLS];
#pragma unroll
    for (int t = 0; t < LZ_COLS; ++t) acc[t] = A(0);
    const int cols = min(LZ_COLS, p.k - g);   // basis columns of this sweep
    const double* col[LZ_COLS];
#pragma unroll
    for (int t = 0; t < LZ_COLS; ++t) col[t] = p.V + (long long)(g + (t < cols ? t : 0)) * p.ldq;
    if (cols == LZ_COLS) {
#pragma unroll 2
      for (long long i = i0; i < p.n; i += step) {
        double v[LZ_COLS];
#pragma unroll
        for (int t = 0; t < LZ_COLS; ++t) v[t] = __ldg(col[t] + i);
        const A ya = lz_in<A>(p.y[i]);
#pragma unroll
        for (int t = 0; t < LZ_COLS; ++t) acc[t] = kc_fma(lz_in<A>(v[t]), ya, acc[t]);
      }
    } else {
      for (long long i = i0; i < p.n; i += step) {
        double v[LZ_COLS];
#pragma unroll
        for (int t = 0; t < LZ_COLS; ++t) v[t] = t < cols ? __ldg(col[t] + i) : 0.0;
        const A ya = lz_in<A>(p.y[i]);
#pragma unroll
        for (int t = 0; t < LZ_COLS; ++t) {
          if (t < cols) acc[t] = kc_fma(lz_in<A>(v[t]), ya, acc[t]);
          else if (t == cols) acc[t] = kc_fma(ya, ya, acc[t]);
        }
      }
    }
    // exchange halves: lane bits 4, 3, 2 choose the column a lane ends with
#pragma unroll
    for (int h = LZ_COLS / 2, m = 16; h >= 1; h >>= 1, m >>= 1)
#pragma unroll
      for (int t = 0; t < h; ++t) {
        const bool up = (lane & m) != 0;
        const A keep = up ? acc[t + h] : acc[t];
        const A give = up ? acc[t] : acc[t + h];
        acc[t] = keep + lz_xor(give, m);
      }
    A r = acc[0];
    r = r + lz_xor(r, 2);
    r = r + lz_xor(r, 1);
    if ((lane & 3) == 0) sh[warp][((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)] = to_d<A>(r);
    __syncthreads();
    if (threadIdx.x < LZ_COLS && g + (int)threadIdx.x <= p.k) {
      double v = 0.0;
#pragma unroll
      for (int u = 0; u < LZ_WARPS; ++u) v += sh[u][threadIdx.x];
      __stcg(p.partial + (long long)(g + threadIdx.x) * gridDim.x + blockIdx.x, v);
    }
    __syncthreads();
  }
}

// c[col] = sum over the blocks of partial[col], col < ncol, in every block's
// shared memory.  Large grids: block b adds columns b, b + grid, .. first.
__device__ __forceinline__ void lz_columns(const LzStep& p, int ncol, double* coef, double* c, unsigned& round) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool direct = (int)gridDim.x <= LZ_DIRECT;
  const int first = direct ? warp : (int)blockIdx.x + (int)gridDim.x * warp;
  const int step = direct ? LZ_WARPS : (int)gridDim.x * LZ_WARPS;
  for (int col = first; col < ncol; col += step) {
    double v = 0.0;
    for (int i = lane; i < (int)gridDim.x; i += 32) v += __ldcg(p.partial + (long long)col * gridDim.x + i);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) {
      if (direct) c[col] = v;
      else __stcg(coef + col, v);
    }
  }
  if (!direct) {
    grid_sync(p.bar, round, p.err);
    for (int col = threadIdx.x; col < ncol; col += LZ_THREADS) c[col] = __ldcg(coef + col);
  }
  __syncthreads();
}

// y -= V c; returns this thread's part of |y|^2.
template <typename A>
__device__ __forceinline__ A lz_update(const LzStep& p, const double* c, A* cs, long long i0, long long step) {
  for (int j = threadIdx.x; j < p.k; j += LZ_THREADS) cs[j] = lz_in<A>(-c[j]);
  __syncthreads();
  A nrm = A(0);
#pragma unroll 2
  for (long long i = i0; i < p.n; i += step) {
    A v = lz_in<A>(p.y[i]);
    const double* q = p.V + i;
    int j = 0;
    for (; j + LZ_COLS <= p.k; j += LZ_COLS) {
      double x[LZ_COLS];
#pragma unroll
      for (int t = 0; t < LZ_COLS; ++t) x[t] = __ldg(q + (long long)(j + t) * p.ldq);
#pragma unroll
      for (int t = 0; t < LZ_COLS; ++t) v = kc_fma(cs[j + t], lz_in<A>(x[t]), v);
    }
    for (; j < p.k; ++j) v = kc_fma(cs[j], lz_in<A>(__ldg(q + (long long)j * p.ldq)), v);
    p.y[i] = to_d<A>(v);
    nrm = kc_fma(v, v, nrm);
  }
  return nrm;
}

// The last block to leave zeroes the counters for the next launch.
__device__ __forceinline__ void lz_leave(const LzStep& p, double alpha, double nrm2) {
  if (threadIdx.x == 0) {
    if (blockIdx.x == 0) {
      *p.alpha_j = alpha;
      *p.beta_j = sqrt(fmax(nrm2, 0.0));
    }
    if (atomicAdd(p.bar + 1, 1u) == gridDim.x - 1) {
      p.bar[0] = 0u;
      p.bar[1] = 0u;
    }
  }
}

// ---- short vectors: the basis columns are shared out as well
// (a step at n = 5104 with 1-46 vectors: 25-55 us in the long form, 22 here)
// Block (rb, cg) of row_blocks x column_groups: rows rb * 256 .., column sweeps
// cg, cg + column_groups, ..  A short vector leaves a thread a row or two, so
// the time is the number of trips to L2 one after another; here a dot phase is
// one sweep per block, and four lanes share a row of an update.
// part[rb * (k + 1) + col]; `w` gives w' (or y) of a row.
template <typename A, typename Row>
__device__ __forceinline__ void lz_short_dots(const LzStep& p, int rb, int row_blocks, int cg, int column_groups,
                                              double (*sh)[LZ_COLS], Row row) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int g = cg * LZ_COLS; g <= p.k; g += column_groups * LZ_COLS) {
    A acc[LZ_COLS];
#pragma unroll
    for (int t = 0; t < LZ_COLS; ++t) acc[t] = A(0);
    for (long long i = (long long)rb * LZ_THREADS + threadIdx.x; i < p.n; i += (long long)row_blocks * LZ_THREADS) {
      double v[LZ_COLS];
#pragma unroll
      for (int t = 0; t < LZ_COLS; ++t) v[t] = g + t < p.k ? __ldg(p.V + (long long)(g + t) * p.ldq + i) : 0.0;
      const A ya = lz_in<A>(row(i));
#pragma unroll
      for (int t = 0; t < LZ_COLS; ++t) {
        if (g + t < p.k) acc[t] = kc_fma(lz_in<A>(v[t]), ya, acc[t]);
        else if (g + t == p.k) acc[t] = kc_fma(ya, ya, acc[t]);
      }
    }
#pragma unroll
    for (int h = LZ_COLS / 2, m = 16; h >= 1; h >>= 1, m >>= 1)
#pragma unroll
      for (int t = 0; t < h; ++t) {
        const bool up = (lane & m) != 0;
        const A keep = up ? acc[t + h] : acc[t];
        const A give = up ? acc[t] : acc[t + h];
        acc[t] = keep + lz_xor(give, m);
      }
    A r = acc[0];
    r = r + lz_xor(r, 2);
    r = r + lz_xor(r, 1);
    if ((lane & 3) == 0) sh[warp][((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)] = to_d<A>(r);
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

// c[col] = sum over the row blocks, one thread a column, in every block.
__device__ __forceinline__ void lz_short_columns(const LzStep& p, int ncol, int row_blocks, double* c) {
  if ((int)threadIdx.x < ncol) {
    double v = 0.0;
#pragma unroll 8
    for (int b = 0; b < row_blocks; ++b) v += __ldcg(p.partial + (long long)b * (p.k + 1) + threadIdx.x);
    c[threadIdx.x] = v;
  }
  __syncthreads();
}

// y = row - V c by quads of lanes; returns this thread's part of |y|^2.
template <typename A, typename Row>
__device__ __forceinline__ A lz_short_update(const LzStep& p, const double* c, A* cs, Row row) {
  for (int j = threadIdx.x; j < p.k; j += LZ_THREADS) cs[j] = lz_in<A>(-c[j]);
  __syncthreads();
  const int sub = threadIdx.x & 3;
  const long long quads = (long long)gridDim.x * (LZ_THREADS / 4);
  A nrm = A(0);
  for (long long i0 = 0; i0 < p.n; i0 += quads) {   // uniform trip count: the quads exchange below
    const long long i = i0 + blockIdx.x * (LZ_THREADS / 4) + (threadIdx.x >> 2);
    const bool in = i < p.n;
    const double* q = p.V + (in ? i : 0);
    A v = A(0);
    for (int j = sub; j < p.k; j += 32) {
      double x[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) x[t] = j + 4 * t < p.k ? __ldg(q + (long long)(j + 4 * t) * p.ldq) : 0.0;
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (j + 4 * t < p.k) v = kc_fma(cs[j + 4 * t], lz_in<A>(x[t]), v);
    }
    v = v + lz_xor(v, 1);
    v = v + lz_xor(v, 2);
    if (in && sub == 0) {
      v = lz_in<A>(row(i)) + v;
      p.y[i] = to_d<A>(v);
      nrm = kc_fma(v, v, nrm);
    }
  }
  return nrm;
}

template <bool FF>
__global__ void __launch_bounds__(LZ_THREADS, 3) lz_short_kernel(LzStep p, int row_blocks, int column_groups) {
  using A = typename std::conditional<FF, ff, double>::type;
  __shared__ double sh[LZ_WARPS][LZ_COLS];
  __shared__ double c[LZ_MAX_K + 4];
  __shared__ A cs[LZ_MAX_K];
  double* red = &sh[0][0];
  unsigned round = 0;
  const int rb = blockIdx.x % row_blocks, cg = blockIdx.x / row_blocks;
  const double* vj = p.V + (long long)(p.k - 1) * p.ldq;
  const double* vp = vj - p.ldq;
  double* part_a = p.partial + (long long)(LZ_MAX_K + 1) * row_blocks;
  double* part_b = part_a + gridDim.x;
  if (cg == 0) {
    double a = 0.0;
    for (long long i = (long long)rb * LZ_THREADS + threadIdx.x; i < p.n; i += (long long)row_blocks * LZ_THREADS)
      a = fma(__ldg(vj + i), __ldcg(p.y + i), a);
    a = lz_block_sum<double>(a, red);
    if (threadIdx.x == 0) __stcg(part_a + rb, a);
  }
  grid_sync(p.bar, round, p.err);
  const double alpha = lz_grid_sum(part_a, row_blocks, red);
  const double beta = p.k >= 2 ? *p.beta_prev : 0.0;
  // w' of a row, formed wherever it is needed: y is written in the update only
  auto residual = [&](long long i) {
    double v = fma(-alpha, __ldg(vj + i), __ldcg(p.y + i));
    return p.k >= 2 ? fma(-beta, __ldg(vp + i), v) : v;
  };
  lz_short_dots<A>(p, rb, row_blocks, cg, column_groups, sh, residual);
  grid_sync(p.bar, round, p.err);
  lz_short_columns(p, p.k + 1, row_blocks, c);
  const double before = c[p.k];
  A t = lz_short_update<A>(p, c, cs, residual);
  double s = lz_block_sum<A>(t, red);
  if (threadIdx.x == 0) __stcg(part_b + blockIdx.x, s);
  grid_sync(p.bar, round, p.err);
  double nrm2 = lz_grid_sum(part_b, gridDim.x, red);
  if (nrm2 < p.ratio * before) {
    auto plain = [&](long long i) { return __ldcg(p.y + i); };
    lz_short_dots<A>(p, rb, row_blocks, cg, column_groups, sh, plain);
    grid_sync(p.bar, round, p.err);
    lz_short_columns(p, p.k, row_blocks, c);
    t = lz_short_update<A>(p, c, cs, plain);
    s = lz_block_sum<A>(t, red);
    if (threadIdx.x == 0) __stcg(part_a + blockIdx.x, s);
    grid_sync(p.bar, round, p.err);
    nrm2 = lz_grid_sum(part_a, gridDim.x, red);
  }
  const double inv = 1.0 / sqrt(nrm2);
  for (long long i = blockIdx.x * (long long)LZ_THREADS + threadIdx.x; i < p.n; i += (long long)gridDim.x * LZ_THREADS)
    p.v_next[i] = __ldcg(p.y + i) * inv;
  lz_leave(p, alpha, nrm2);
}

template <bool FF>
__global__ void __launch_bounds__(LZ_THREADS, 3) lz_step_kernel(LzStep p) {
  using A = typename std::conditional<FF, ff, double>::type;
  __shared__ double sh[LZ_WARPS][LZ_COLS];
  __shared__ double c[LZ_MAX_K + 4];
  __shared__ A cs[LZ_MAX_K];
  double* red = &sh[0][0];
  unsigned round = 0;
  const long long i0 = blockIdx.x * (long long)LZ_THREADS + threadIdx.x;
  const long long step = (long long)gridDim.x * LZ_THREADS;
  const double* vj = p.V + (long long)(p.k - 1) * p.ldq;
  const double* vp = vj - p.ldq;
  // two partial-sum regions that scalars use in turn
  double* part_a = p.partial + (long long)(LZ_MAX_K + 1) * gridDim.x;
  double* part_b = part_a + gridDim.x;
  // alpha_j = v_j . y
  double a = 0.0;
  for (long long i = i0; i < p.n; i += step) a = fma(__ldg(vj + i), p.y[i], a);
  a = lz_block_sum<double>(a, red);
  if (threadIdx.x == 0) __stcg(part_a + blockIdx.x, a);
  grid_sync(p.bar, round, p.err);
  const double alpha = lz_grid_sum(part_a, gridDim.x, red);
  // w' = y - alpha_j v_j - beta_{j-1} v_{j-1}
  const double beta = p.k >= 2 ? *p.beta_prev : 0.0;
  for (long long i = i0; i < p.n; i += step) {
    double v = fma(-alpha, __ldg(vj + i), p.y[i]);
    if (p.k >= 2) v = fma(-beta, __ldg(vp + i), v);
    p.y[i] = v;
  }
  lz_dots<A>(p, sh, i0, step);
  grid_sync(p.bar, round, p.err);
  lz_columns(p, p.k + 1, p.coef, c, round);
  const double before = c[p.k];
  A t = lz_update<A>(p, c, cs, i0, step);
  double s = lz_block_sum<A>(t, red);
  if (threadIdx.x == 0) __stcg(part_b + blockIdx.x, s);
  grid_sync(p.bar, round, p.err);
  double nrm2 = lz_grid_sum(part_b, gridDim.x, red);
  if (nrm2 < p.ratio * before) {
    lz_dots<A>(p, sh, i0, step);
    grid_sync(p.bar, round, p.err);
    lz_columns(p, p.k, p.coef, c, round);
    t = lz_update<A>(p, c, cs, i0, step);
    s = lz_block_sum<A>(t, red);
    if (threadIdx.x == 0) __stcg(part_a + blockIdx.x, s);
    grid_sync(p.bar, round, p.err);
    nrm2 = lz_grid_sum(part_a, gridDim.x, red);
  }
  const double inv = 1.0 / sqrt(nrm2);
  for (long long i = i0; i < p.n; i += step) p.v_next[i] = p.y[i] * inv;
  lz_leave(p, alpha, nrm2);
}

}  // namespace

// Vectors of up to 16384 rows: a row per thread in the dots, the column sweeps
// on further blocks.  Longer ones: two rows a thread up to the resident maximum.
int launch_lz_step(const LzStep& p, int ff_arith, cudaStream_t s) {
  if (p.k < 1 || p.k > LZ_MAX_K) return -7;
  const bool is_short = p.n <= 64 * LZ_THREADS;
  const void* kern = is_short ? (ff_arith ? (const void*)lz_short_kernel<true> : (const void*)lz_short_kernel<false>)
                              : (ff_arith ? (const void*)lz_step_kernel<true> : (const void*)lz_step_kernel<false>);
  static int resident[4] = {0, 0, 0, 0};
  int& cap = resident[(ff_arith ? 1 : 0) + (is_short ? 2 : 0)];
  if (!cap) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, LZ_THREADS, 0);
    cap = std::max(1, std::min(kLzMaxBlocks, std::min(3, per) * sms));
  }
  LzStep arg = p;
  int row_blocks = (int)std::min<long long>(std::min(64, cap), (p.n + LZ_THREADS - 1) / LZ_THREADS);
  int column_groups = std::max(1, std::min(cap / row_blocks, (p.k + LZ_COLS) / LZ_COLS));
  const long long want = (p.n + 2 * LZ_THREADS - 1) / (2 * LZ_THREADS);
  const int blocks = is_short ? row_blocks * column_groups : (int)std::max(1LL, std::min<long long>(cap, want));
  void* args[] = {&arg, &row_blocks, &column_groups};
  if (cudaLaunchCooperativeKernel(kern, dim3(blocks), dim3(LZ_THREADS), args, 0, s) != cudaSuccess) return -3;
  count_launches(1);
  return 0;
}

}  // namespace qed
