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

// Sum of one value per block, in block order by lanes; valid in every thread.
__device__ __forceinline__ double lz_grid_sum(const double* part, double* red) {
  if (threadIdx.x < 32) {
    double v = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += 32) v += __ldcg(part + i);
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
  const double alpha = lz_grid_sum(part_a, red);
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
  double nrm2 = lz_grid_sum(part_b, red);
  if (nrm2 < p.ratio * before) {
    lz_dots<A>(p, sh, i0, step);
    grid_sync(p.bar, round, p.err);
    lz_columns(p, p.k, p.coef, c, round);
    t = lz_update<A>(p, c, cs, i0, step);
    s = lz_block_sum<A>(t, red);
    if (threadIdx.x == 0) __stcg(part_a + blockIdx.x, s);
    grid_sync(p.bar, round, p.err);
    nrm2 = lz_grid_sum(part_a, red);
  }
  const double inv = 1.0 / sqrt(nrm2);
  for (long long i = i0; i < p.n; i += step) p.v_next[i] = p.y[i] * inv;
  if (threadIdx.x == 0) {
    if (blockIdx.x == 0) {
      *p.alpha_j = alpha;
      *p.beta_j = sqrt(fmax(nrm2, 0.0));
    }
    // the last block to leave zeroes the counters for the next launch
    if (atomicAdd(p.bar + 1, 1u) == gridDim.x - 1) {
      p.bar[0] = 0u;
      p.bar[1] = 0u;
    }
  }
}

}  // namespace

// Blocks: two rows a thread while that leaves SMs idle (small problems are
// latency-bound), the resident maximum for large ones.
int launch_lz_step(const LzStep& p, int ff_arith, cudaStream_t s) {
  if (p.k < 1 || p.k > LZ_MAX_K) return -7;
  auto kern = ff_arith ? lz_step_kernel<true> : lz_step_kernel<false>;
  static int resident[2] = {0, 0};
  int& cap = resident[ff_arith ? 1 : 0];
  if (!cap) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, LZ_THREADS, 0);
    cap = std::max(1, std::min(kLzMaxBlocks, std::min(3, per) * sms));
  }
  const long long want = (p.n + 2 * LZ_THREADS - 1) / (2 * LZ_THREADS);
  const int blocks = (int)std::max(1LL, std::min<long long>(cap, want));
  LzStep arg = p;
  void* args[] = {&arg};
  if (cudaLaunchCooperativeKernel((const void*)kern, dim3(blocks), dim3(LZ_THREADS), args, 0, s) != cudaSuccess)
    return -3;
  count_launches(1);
  return 0;
}

}  // namespace qed
