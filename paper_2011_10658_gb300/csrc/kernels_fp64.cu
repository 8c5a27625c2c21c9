// FP64 SIMT kernels: grouped K-concatenated GEMM with optional row gathers,
// Lanczos vector reductions, per-sector Cholesky, tridiagonal eigensolver.
// GB300's FP64 rate is a small fraction of its tensor throughput, so these
// kernels are simple register-tiled DFMA loops; the mixed-precision path
// replaces the hot contraction with tensor-core kernels.
#include <cfloat>
#include <atomic>
#include <type_traits>
#include <cstdio>
#include <mutex>
#include <set>
#include <utility>

#include "ffloat.cuh"
#include "kernels.cuh"

namespace qed {

static std::atomic<long long> g_launches{0};
long long launch_count() { return g_launches.load(); }
void count_launches(int n) { g_launches += n; }

void allow_smem(const void* kern, int bytes) {
  static std::mutex lock;
  static std::set<std::pair<int, const void*>> done;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> guard(lock);
  if (done.insert({dev, kern}).second) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

namespace {

constexpr int BK = 16;
constexpr int THREADS = 256;

// Two-level index e -> (e / in) * outer + (e % in) * inner (in = 0: one level).
__device__ __forceinline__ long long two_level(int e, int in, unsigned div, long long inner, long long outer) {
  if (in == 0) return (long long)e * inner;
  const int o = in == 1 ? e : (int)__umulhi((unsigned)e, div);
  return (long long)o * outer + (long long)(e - o * in) * inner;
}

// Row maps are sign-encoded: -1 = zero row, otherwise (row << 1) | negate.
// Arithmetic in T (FP64, or FP32 with the operands converted first).
template <typename T>
__device__ __forceinline__ T load_a(const KChunk& c, int m, int k) {
  long long row = m;
  T scale = T(1);
  if (c.amap) {
    int r = c.amap[m];
    if (r < 0) return T(0);
    row = r >> 1;
    if (r & 1) scale = T(-1);
  }
  if (c.aval) scale *= to_t<T>(c.aval[m]);
  return scale * to_t<T>(c.A[row * c.a_m + two_level(k, c.kin, c.kdiv, c.a_k, c.a_ko)]);
}

template <typename T>
__device__ __forceinline__ T load_b(const KChunk& c, int k, long long n_off) {
  if (!c.bmap) return to_t<T>(c.B[two_level(k, c.kin, c.kdiv, c.b_k, c.b_ko) + n_off]);
  const int r = c.bmap[k];
  if (r < 0) return T(0);
  T scale = (r & 1) ? T(-1) : T(1);
  if (c.bval) scale *= to_t<T>(c.bval[k]);
  return scale * to_t<T>(c.B[(long long)(r >> 1) * c.b_k + n_off]);
}

// One CTA computes a BM x BN tile of one output (16 x 16 threads, each a
// BM/16 x BN/16 register tile) over its chunk range, K staged in slabs of 16.
template <typename T, int BM, int BN>
__global__ void __launch_bounds__(THREADS) kc_gemm_kernel(const KTile* __restrict__ tiles,
                                                           const KOutput* __restrict__ outs,
                                                           const KChunk* __restrict__ chunks,
                                                           double* __restrict__ scratch) {
  constexpr int TM = BM / 16, TN = BN / 16;
  __shared__ T As[BK][BM + 1];
  __shared__ T Bs[BK][BN + 1];
  const KTile tile = tiles[blockIdx.x];
  const KOutput out = outs[tile.out];
  const int tid = threadIdx.x;
  const int tx = tid % 16, ty = tid / 16;
  T acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = T(0);
  for (int ci = tile.chunk_begin; ci < tile.chunk_end; ++ci) {
    const KChunk c = chunks[ci];
    if (c.add) {
      // C[m,n] += alpha * A[m,n]
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          const int m = tile.m0 + ty * TM + i, n = tile.n0 + tx * TN + j;
          if (m < out.M && n < out.N) acc[i][j] += raw_t<T>(c.alpha) * load_a<T>(c, m, n);
        }
      continue;
    }
    const T alpha = raw_t<T>(c.alpha);
    for (int k0 = 0; k0 < c.K; k0 += BK) {
      for (int e = tid; e < BM * BK; e += THREADS) {
        const int mm = e / BK, kk = e % BK;
        const int m = tile.m0 + mm, k = k0 + kk;
        As[kk][mm] = (m < out.M && k < c.K) ? alpha * load_a<T>(c, m, k) : T(0);
      }
      for (int e = tid; e < BN * BK; e += THREADS) {
        const int kk = e / BN, nn = e % BN;
        const int n = tile.n0 + nn, k = k0 + kk;
        Bs[kk][nn] = (n < out.N && k < c.K) ? load_b<T>(c, k, two_level(n, out.nin, out.ndiv, c.b_n, c.b_no)) : T(0);
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        T a[TM], bv[TN];
#pragma unroll
        for (int i = 0; i < TM; ++i) a[i] = As[kk][ty * TM + i];
#pragma unroll
        for (int j = 0; j < TN; ++j) bv[j] = Bs[kk][tx * TN + j];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[i][j] = kc_fma(a[i], bv[j], acc[i][j]);
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int m = tile.m0 + ty * TM + i, n = tile.n0 + tx * TN + j;
      if (m >= out.M || n >= out.N) continue;
      const double v = to_d<T>(acc[i][j]);
      if (tile.part >= 0) {
        scratch[out.part_off + (long long)tile.part * out.M * out.N + (long long)m * out.N + n] = v;
      } else {
        double* p = out.C + (long long)m * out.c_m + two_level(n, out.nin, out.ndiv, out.c_n, out.c_no);
        *p = out.accumulate ? (*p + v) : v;
      }
    }
}

__global__ void kc_reduce_kernel(const KOutput* __restrict__ outs, const int* __restrict__ red_list,
                                 const double* __restrict__ scratch) {
  const KOutput out = outs[red_list[blockIdx.y]];
  const long long mn = (long long)out.M * out.N;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < mn; e += (long long)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int p = 0; p < out.n_parts; ++p) s += scratch[out.part_off + p * mn + e];
    int m = (int)(e / out.N), n = (int)(e % out.N);
    double* c = out.C + (long long)m * out.c_m + two_level(n, out.nin, out.ndiv, out.c_n, out.c_no);
    *c = out.accumulate ? (*c + s) : s;
  }
}

// ------------------------------------------------------------ reductions
constexpr int RED_THREADS = 256;
constexpr int RED_BLOCKS = 304;   // 2 x 152 SMs

__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[RED_THREADS / 32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x < 32) {
    r = threadIdx.x < RED_THREADS / 32 ? sh[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  }
  return r;   // valid in thread 0
}

__global__ void dot_partial_kernel(const double* __restrict__ x, const double* __restrict__ y, long long n,
                                   double* __restrict__ partial) {
  double v = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    v = fma(x[i], y[i], v);
  v = block_sum(v);
  if (threadIdx.x == 0) partial[blockIdx.x] = v;
}

__global__ void finish_kernel(const double* __restrict__ partial, int count, double* __restrict__ out) {
  double v = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) v += partial[i];
  v = block_sum(v);
  if (threadIdx.x == 0) out[0] = v;
}

__global__ void combine_kernel(const double* __restrict__ Q, long long ldq, int k, const double* __restrict__ c,
                               double* __restrict__ x, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    double v = 0.0;
    for (int j = 0; j < k; ++j) v = fma(c[j], Q[(long long)j * ldq + i], v);
    x[i] = v;
  }
}

__global__ void sqrt_kernel(const double* in, double* out) {
  if (threadIdx.x == 0 && blockIdx.x == 0) out[0] = sqrt(fmax(in[0], 0.0));
}

__global__ void axpby_kernel(const double* __restrict__ x, double* __restrict__ y, long long n, const double* a_dev,
                             double a_const, double a_sign, const double* b_dev, double b_const) {
  const double a = a_sign * (a_dev ? *a_dev : a_const);
  const double b = b_dev ? *b_dev : b_const;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = fma(a, x[i], b * y[i]);
}

__global__ void scale_inv_sqrt_kernel(const double* __restrict__ x, double* __restrict__ y, long long n,
                                      const double* nrm2, const int* gate) {
  if (gate && *gate) return;
  const double inv = 1.0 / sqrt(*nrm2);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = x[i] * inv;
}

__global__ void copy_kernel(const double* __restrict__ x, double* __restrict__ y, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = x[i];
}

__global__ void add_scaled_kernel(const double* __restrict__ x, double* __restrict__ y, long long n, double a) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = fma(a, x[i], y[i]);
}

// y[i] = sum of x[r * n + i] over the rows r.
__global__ void sum_rows_kernel(const double* __restrict__ x, long long n, int rows, double* __restrict__ y) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    double v = 0.0;
    for (int r = 0; r < rows; ++r) v += x[r * n + i];
    y[i] = v;
  }
}

__global__ void zero_kernel(double* __restrict__ x, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    x[i] = 0.0;
}

// flag = 1 if some x[i] is NaN or infinite (exponent field all ones).
__global__ void check_finite_kernel(const double* __restrict__ x, long long n, int* flag) {
  bool bad = false;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    bad |= ((__double_as_longlong(x[i]) >> 52) & 0x7ff) == 0x7ff;
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicExch(flag, 1);
}

__global__ void to_float_kernel(const double* __restrict__ x, float* __restrict__ y, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = (float)x[i];
}

__global__ void to_double_kernel(const float* __restrict__ x, double* __restrict__ y, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = (double)x[i];
}

// SplitMix64 (Steele, Lea & Flood 2014), counter form: output i (1-based)
// is mix(seed + i * gamma); value 2 * (x >> 11) * 2^-53 - 1.
__global__ void fill_uniform_kernel(double* __restrict__ x, long long n, uint64_t seed, uint64_t start) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    uint64_t z = seed + (start + (uint64_t)i + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z = z ^ (z >> 31);
    x[i] = 2.0 * (double)(z >> 11) * 0x1.0p-53 - 1.0;
  }
}

// Upper Cholesky G = R^T R and X = R^{-1}, one CTA per matrix, in one n x n
// array of shared memory: R above the diagonal (its diagonal in rd), X
// transposed below it.  Bound by the serial chain (an FP64 operation takes 65
// cycles and more here): a square root, a division and an update per column of
// R, then n (n - 1) / 2 multiply-adds and n divisions down the last column of
// X.  Every thread that divides by a diagonal takes its square root itself,
// which saves a barrier per column.  The order of the operations is part of
// the result: centre moves feed gauges and low-precision updates that turn a
// changed last place into a visible difference, so the root-free form with X
// grown by outer products (32 us a launch of sectors up to 32 columns; this form
// 53, with X in global memory 64) is not used.
__global__ void __launch_bounds__(256) cholesky_inv_kernel(double* G, double* Rinv, const long long* off,
                                                           const int* nn, const int* ldd, int* status,
                                                           double ill_cond) {
  extern __shared__ double sh[];
  const int idx = blockIdx.x;
  const int n = nn[idx], ld = ldd[idx], lr = n | 1;
  double* g = G + off[idx];
  double* ri = Rinv + off[idx];
  double* R = sh;              // n rows of lr
  __shared__ double rd[160], xd[160], gmax;
  __shared__ int bad;
  const int tid = threadIdx.x;
  for (int e = tid; e < n * n; e += blockDim.x) R[(e / n) * lr + e % n] = g[(e / n) * ld + (e % n)];
  if (tid == 0) bad = 0;
  __syncthreads();
  // largest original diagonal = squared largest column norm of the factored matrix
  if (tid < 32) {
    double mx = 0.0;
    for (int j = tid; j < n; j += 32) mx = fmax(mx, R[j * lr + j]);
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (tid == 0) gmax = mx;
  }
  __syncthreads();
  // row j divided by r_jj = sqrt(g_jj), then trailing g_ab -= r_ja r_jb
  for (int j = 0; j < n; ++j) {
    const int w = n - j - 1;
    if (tid < w || tid == 0) {
      double d = R[j * lr + j];
      if (!(d > 0.0)) {
        if (tid == 0) bad = 1;
        d = 1.0;
      } else if (tid == 0 && d <= ill_cond * gmax) {
        bad = bad ? bad : 2;
      }
      const double r = sqrt(d);
      if (tid == 0) rd[j] = r;
      if (tid < w) R[j * lr + j + 1 + tid] /= r;
    }
    __syncthreads();
    for (int e = tid; e < w * w; e += blockDim.x) {
      const int a = j + 1 + e / w, b = j + 1 + e % w;
      if (b >= a) R[a * lr + b] = fma(-R[j * lr + a], R[j * lr + b], R[a * lr + b]);
    }
    __syncthreads();
  }
  for (int e = tid; e < n * n; e += blockDim.x) {
    const int a = e / n, b = e - a * n;
    g[a * ld + b] = b > a ? R[a * lr + b] : (b == a ? rd[a] : 0.0);
  }
  __syncthreads();   // below the diagonal X is written from here on
  // R X = I, a column per thread, from the diagonal up
  if (tid < n) {
    double* x = R + tid * lr;   // X of column tid
    const double xc = 1.0 / rd[tid];
    xd[tid] = xc;
    for (int a = tid - 1; a >= 0; --a) {
      const double* r = R + a * lr;
      double v = 0.0;
#pragma unroll 4
      for (int b = a + 1; b < tid; ++b) v = fma(-r[b], x[b], v);
      v = fma(-r[tid], xc, v);
      x[a] = v / rd[a];
    }
  }
  __syncthreads();
  for (int e = tid; e < n * n; e += blockDim.x) {
    const int a = e / n, b = e - a * n;
    ri[a * ld + b] = b > a ? R[b * lr + a] : (b == a ? xd[a] : 0.0);
  }
  if (tid == 0) status[idx] = bad;
}


// Classical Gram-Schmidt applied twice per column, one CTA per sector matrix
// (column-major m x n at X + xoff, Q written in place, R (n x n) at
// R + roff with leading dimension ldr).  A column whose remainder is at
// most dep_tol * (largest column norm) is dependent: R_jj = 0 and q_j is
// the first unit vector e_k (k increasing, never reused) whose remainder
// after two projections exceeds accept.
constexpr int QR_THREADS = 1024;

__device__ double cta_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  if (w == 0) {
    double r = l < (int)(blockDim.x / 32) ? red[l] : 0.0;
    for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    if (l == 0) red[32] = r;
  }
  __syncthreads();
  return red[32];
}

// c[i] = <q_i, v> for i < j (warp per i), then v -= sum_i c[i] q_i.
__device__ void project_out(const double* X, long long m, int j, double* v, double* c, double* Rcol) {
  const int w = threadIdx.x / 32, l = threadIdx.x % 32, nw = blockDim.x / 32;
  for (int i = w; i < j; i += nw) {
    const double* q = X + (long long)i * m;
    double acc = 0.0;
    for (long long r = l; r < m; r += 32) acc = fma(q[r], v[r], acc);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (l == 0) c[i] = acc;
  }
  __syncthreads();
  for (long long r = threadIdx.x; r < m; r += blockDim.x) {
    double a = v[r];
    for (int i = 0; i < j; ++i) a = fma(-c[i], X[(long long)i * m + r], a);
    v[r] = a;
  }
  if (Rcol)
    for (int i = threadIdx.x; i < j; i += blockDim.x) Rcol[i] += c[i];
  __syncthreads();
}

__global__ void __launch_bounds__(QR_THREADS) cgs2_qr_kernel(double* X, const long long* xoff, const int* rows,
                                                              const int* cols, double* R, const long long* roff,
                                                              int ldr, double dep_tol, double accept) {
  __shared__ double red[40];
  __shared__ double c[256];
  __shared__ double rcol[256];
  const int sidx = blockIdx.x;
  const long long m = rows[sidx];
  const int n = cols[sidx];
  double* x = X + xoff[sidx];
  double* Rs = R + roff[sidx];
  double scale = 0.0;
  for (int j = 0; j < n; ++j) {
    double acc = 0.0;
    for (long long r = threadIdx.x; r < m; r += blockDim.x) acc = fma(x[j * m + r], x[j * m + r], acc);
    scale = fmax(scale, sqrt(cta_sum(acc, red)));
  }
  long long next_k = 0;
  for (int j = 0; j < n; ++j) {
    double* v = x + (long long)j * m;
    for (int i = threadIdx.x; i < n; i += blockDim.x) rcol[i] = 0.0;
    __syncthreads();
    project_out(x, m, j, v, c, rcol);
    project_out(x, m, j, v, c, rcol);
    double acc = 0.0;
    for (long long r = threadIdx.x; r < m; r += blockDim.x) acc = fma(v[r], v[r], acc);
    const double nv = sqrt(cta_sum(acc, red));
    if (nv > dep_tol * scale) {
      const double inv = 1.0 / nv;
      for (long long r = threadIdx.x; r < m; r += blockDim.x) v[r] *= inv;
      if (threadIdx.x == 0) rcol[j] = nv;
    } else {
      if (threadIdx.x == 0) rcol[j] = 0.0;
      // completion by unit vectors
      for (; next_k < m; ++next_k) {
        for (long long r = threadIdx.x; r < m; r += blockDim.x) v[r] = (r == next_k) ? 1.0 : 0.0;
        __syncthreads();
        project_out(x, m, j, v, c, nullptr);
        project_out(x, m, j, v, c, nullptr);
        double a2 = 0.0;
        for (long long r = threadIdx.x; r < m; r += blockDim.x) a2 = fma(v[r], v[r], a2);
        const double nw = sqrt(cta_sum(a2, red));
        if (nw > accept) {
          const double inv = 1.0 / nw;
          for (long long r = threadIdx.x; r < m; r += blockDim.x) v[r] *= inv;
          ++next_k;
          break;
        }
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) Rs[(long long)i * ldr + j] = i <= j ? rcol[i] : 0.0;
    __syncthreads();
  }
}

// ------------------------------------------------------------ tridiagonal
// Lowest eigenpair of the k x k symmetric tridiagonal T (diagonal a, squared
// off-diagonal b2) of a Lanczos cycle.  The leading principal minors
// p_i(x) = det(T_i - x I) obey p_i = (a_i - x) p_{i-1} - b2_{i-1} p_{i-2};
// the number of sign changes along p_0 = 1, p_1, .., p_k is the number of
// eigenvalues below x (Sturm).  Every operation is a multiply-add, so a warp
// evaluates 32 counts at once; the state is rescaled by exact powers of two.
constexpr int TRI_MAX = 128;
constexpr int RESTART_MAX = 8;   // Ritz vectors kept by a thick restart

__device__ __forceinline__ int dexp(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// exact rescaling of the recurrence state (p, pm[, d, dm]) by 2^-512 / 2^512
__device__ __forceinline__ void rescale2(double& p, double& pm) {
  const int e = dexp(p);
  if (e > 1023 + 512) {
    p *= 0x1p-512; pm *= 0x1p-512;
  } else if (e < 1023 - 512 && dexp(pm) < 1023 - 512) {
    p *= 0x1p+512; pm *= 0x1p+512;
  }
}

__device__ int sturm_minors(const double* a, const double* b2, int k, double x) {
  double pm = 1.0, p = a[0] - x;
  int neg = __double2hiint(p) < 0 && p != 0.0;
  int cnt = neg;
  for (int i = 1; i < k; ++i) {
    const double pn = fma(a[i] - x, p, -b2[i - 1] * pm);
    const int nn = __double2hiint(pn) < 0 && pn != 0.0;   // zero counts as positive
    cnt += nn ^ neg;
    neg = nn;
    pm = p;
    p = pn;
    rescale2(p, pm);
  }
  return cnt;
}

// Eigenvector of T for the eigenvalue theta by inverse iteration with a shift
// just below theta, one warp: tridiagonal LU (Thomas) once, then solves.  Every
// chain (elimination, substitution, a dot product) is one FP64 latency per row
// in lane 0, the rest is one row per lane.  cp, inv: the factors (k doubles of
// shared memory each), x the vector.
__device__ void inverse_lu(const double* a, const double* b, int k, double theta, double scale, double* cp,
                           double* inv) {
  const double shift = theta - 1e-13 * fmax(scale, 1e-300) - 1e-300;
  if ((threadIdx.x & 31) == 0) {
    double denom = a[0] - shift;
    if (denom == 0.0) denom = 1e-300;
    inv[0] = denom;   // the first row divides
    double c = (k > 1 ? b[0] : 0.0) / denom;
    cp[0] = c;
    for (int i = 1; i < k; ++i) {
      double m = fma(-b[i - 1], c, a[i] - shift);
      if (m == 0.0) m = 1e-300;
      const double r = 1.0 / m;
      c = (i < k - 1 ? b[i] : 0.0) * r;
      cp[i] = c;
      inv[i] = r;
    }
  }
  __syncwarp();
}

__device__ void inverse_solve(const double* b, int k, const double* cp, const double* inv, double* x) {
  if ((threadIdx.x & 31) == 0) {
    double d = x[0] / inv[0];
    x[0] = d;
#pragma unroll 4
    for (int i = 1; i < k; ++i) {
      d = fma(-b[i - 1], d, x[i]) * inv[i];
      x[i] = d;
    }
#pragma unroll 4
    for (int i = k - 2; i >= 0; --i) {
      d = fma(-cp[i], d, x[i]);
      x[i] = d;
    }
  }
  __syncwarp();
}

// sum of x[i] y[i], rows one after another; valid in every lane.
__device__ double chain_dot(const double* x, const double* y, int k) {
  double h = 0.0;
  if ((threadIdx.x & 31) == 0) {
#pragma unroll 8
    for (int i = 0; i < k; ++i) h = fma(x[i], y[i], h);
  }
  return __shfl_sync(0xffffffffu, h, 0);
}

__device__ void remove_along(const double* q, double* x, int k) {
  const double h = chain_dot(q, x, k);
  for (int i = threadIdx.x & 31; i < k; i += 32) x[i] = fma(-h, q[i], x[i]);
  __syncwarp();
}

__device__ void make_unit(double* x, int k) {
  const double inv = 1.0 / sqrt(chain_dot(x, x, k));
  for (int i = threadIdx.x & 31; i < k; i += 32) x[i] *= inv;
  __syncwarp();
}

__device__ void inverse_start(double* x, int k, int n_prev) {
  for (int i = threadIdx.x & 31; i < k; i += 32) x[i] = n_prev == 0 ? 1.0 : 1.0 + 0.37 * (double)(i % (n_prev + 2));
  __syncwarp();
}

constexpr int INV_ITERS = 3;

// The lowest eigenvector: no lower ones to stay orthogonal to, x[0] >= 0.
__device__ void inverse_iteration(const double* a, const double* b, int k, double theta, double scale, double* cp,
                                  double* inv, double* x) {
  inverse_lu(a, b, k, theta, scale, cp, inv);
  inverse_start(x, k, 0);
  for (int it = 0; it < INV_ITERS; ++it) {
    inverse_solve(b, k, cp, inv, x);
    make_unit(x, k);
  }
  const bool flip = x[0] < 0.0;
  __syncwarp();
  if (flip)
    for (int i = threadIdx.x & 31; i < k; i += 32) x[i] = -x[i];
  __syncwarp();
}

// Multisection for the eigenvalue of index idx (0 = lowest) by N threads, of
// which this is thread t: on entry [lo, hi] holds it (count(lo) <= idx <
// count(hi)); each round counts at N interior points, and the bracket shrinks
// (N + 1)-fold, until it is a few ulps wide.  below(above) returns how many of
// the N threads are not above.  All threads return the same bracket.
template <int N, typename Below>
__device__ void multisect(const double* a, const double* b2, int k, int idx, int t, Below below, double& lo,
                          double& hi) {
  for (int round = 0; round < 64; ++round) {
    const double w = hi - lo;
    if (w <= 4.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi)) + 1e-300) break;
    const double x = lo + w * ((double)(t + 1) * (1.0 / (N + 1)));
    const int f = below(sturm_minors(a, b2, k, x) > idx);
    const double nlo = f > 0 ? lo + w * ((double)f * (1.0 / (N + 1))) : lo;
    const double nhi = f < N ? lo + w * ((double)(f + 1) * (1.0 / (N + 1))) : hi;
    if (!(nhi - nlo < w)) break;   // no progress left at this precision
    lo = nlo;
    hi = nhi;
  }
}

struct WarpBelow {
  __device__ int operator()(bool above) const { return 32 - __popc(__ballot_sync(0xffffffffu, above)); }
};
template <int N>
struct BlockBelow {
  __device__ int operator()(bool above) const { return N - __syncthreads_count(above); }
};

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Warp-collective: stage (a, b, b2) of the tridiagonal and 1 / b in shared
// memory and return its Gershgorin bracket (widened) and scale.
__device__ void stage_tridiag(const double* alpha, const double* beta, int k, double* a, double* b, double* b2,
                              double* ib, double& lo, double& hi, double& scale) {
  const int lane = threadIdx.x & 31;
  for (int i = lane; i < k; i += 32) {
    a[i] = alpha[i];
    const double bi = i < k - 1 ? beta[i] : 0.0;
    b[i] = bi;
    b2[i] = bi * bi;
    ib[i] = i < k - 1 ? 1.0 / bi : 0.0;
  }
  __syncwarp();
  lo = 1e300;
  hi = -1e300;
  for (int i = lane; i < k; i += 32) {
    const double r = (i > 0 ? fabs(b[i - 1]) : 0.0) + fabs(b[i]);
    lo = fmin(lo, a[i] - r);
    hi = fmax(hi, a[i] + r);
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  const double span = hi - lo;
  scale = fmax(fabs(lo), fabs(hi));
  lo -= 1e-12 * span + 1e-300;
  hi += 1e-12 * span + 1e-300;
}

// Warp-collective eigenvector of T for the eigenvalue theta, by the three-term
// recurrences from both ends joined where they fit best (the twisted
// factorisation of Parlett and Dhillon): with f running down from f_0 = 1 and
// g up from g_{k-1} = 1, row r of (T - theta) x misses zero by
//   gamma_r = (a_r - theta) + b_{r-1} f_{r-1} / f_r + b_r g_{r+1} / g_r
// when x is f / f_r above r and g / g_r below; r is the row of least |gamma|.
// Lanes 0 and 1 run the two recurrences in step; the rest is parallel.  f, g,
// c1: k, k and 2 k doubles of shared memory; f returns the unit vector.  False
// if no row has a finite gamma (the recurrences left the FP64 range), f then
// undefined.
__device__ bool twisted_vector(const double* a, const double* b, const double* ib, int k, double theta, double* f,
                               double* g, double* c1) {
  const int lane = threadIdx.x & 31;
  for (int i = lane; i < k; i += 32) {
    const double t = theta - a[i];
    c1[i] = t * ib[i];                                // f_{i+1} = c1[i] f_i - (b_{i-1} / b_i) f_{i-1}
    c1[k + k - 1 - i] = i > 0 ? t * ib[i - 1] : 0.0;  // g_{i-1} likewise, stored in running order
  }
  __syncwarp();
  if (lane < 2) {
    const bool down = lane == 0;
    double* out = down ? f : g;
    const double* c = down ? c1 : c1 + k;
    double pm = 0.0, p = 1.0;
    int at = down ? 0 : k - 1;
    const int dir = down ? 1 : -1;
    out[at] = 1.0;
    for (int i = 0; i + 1 < k; ++i) {
      // coupling ratio to the entry before: b_{i-1} / b_i going down
      const int lo = down ? i - 1 : k - 1 - i, hi = down ? i : k - 2 - i;
      const double q = i > 0 ? b[lo] * ib[hi] : 0.0;
      const double pn = fma(c[i], p, -q * pm);
      pm = p;
      p = pn;
      at += dir;
      out[at] = p;
    }
  }
  __syncwarp();
  double best = 1e308;
  int r = -1;
  for (int i = lane; i < k; i += 32) {
    double gm = a[i] - theta;
    if (i > 0) gm += b[i - 1] * (f[i - 1] / f[i]);
    if (i < k - 1) gm += b[i] * (g[i + 1] / g[i]);
    gm = fabs(gm);
    if (gm < best) { best = gm; r = i; }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int orr = __shfl_xor_sync(0xffffffffu, r, o);
    if (orr >= 0 && (ob < best || (ob == best && (r < 0 || orr < r)))) { best = ob; r = orr; }
  }
  if (r < 0) return false;
  const double fi = 1.0 / f[r], gi = 1.0 / g[r];
  __syncwarp();
  double n2 = 0.0;
  for (int i = lane; i < k; i += 32) {
    const double x = i <= r ? f[i] * fi : g[i] * gi;
    f[i] = x;
    n2 = fma(x, x, n2);
  }
  n2 = warp_sum(n2);
  __syncwarp();
  const double inv = 1.0 / sqrt(n2);
  __syncwarp();
  for (int i = lane; i < k; i += 32) f[i] *= inv;
  __syncwarp();
  return isfinite(inv) && n2 >= 1.0;
}

// Four warps (one per scheduler: a warp's FP64 instruction holds its
// scheduler's pipe for 64 cycles, so four warps count at four times the points
// in the same time).  out[0] = theta (lowest eigenvalue), out[1] = |beta[k-1]|
// |s_k| (the Ritz residual estimate).  prev (optional): the lowest Ritz value
// of a smaller basis of the same run, an upper bound of theta; the first round
// then counts at distances from it that halve every second or third point.
// GB300: 12-90 us (k = 1-64); 100 us on average over an FP64 sweep of 2x2x2
// with 32 points a round and inverse iteration.
constexpr int TRI_THREADS = 128;

__global__ void __launch_bounds__(TRI_THREADS) tridiag_lowest_kernel(const double* __restrict__ alpha,
                                                                     const double* __restrict__ beta, int k,
                                                                     double* out, const double* prev) {
  __shared__ double a[TRI_MAX], b[TRI_MAX], b2[TRI_MAX], ib[TRI_MAX];
  __shared__ double f[TRI_MAX], g[TRI_MAX], c1[2 * TRI_MAX], bracket[3];
  const int t = threadIdx.x;
  double lo, hi, scale;
  if (t < 32) {
    stage_tridiag(alpha, beta, k, a, b, b2, ib, lo, hi, scale);
    if (t == 0) { bracket[0] = lo; bracket[1] = hi; bracket[2] = scale; }
  }
  __syncthreads();
  lo = bracket[0];
  hi = bracket[1];
  scale = bracket[2];
  const BlockBelow<TRI_THREADS> below;
  if (prev) {
    const double top = *prev + 4.0 * DBL_EPSILON * scale, w = top - lo;
    if (w > 0.0 && top < hi) {
      // distances w 2^(-55 t / 128) below top; the last point is top itself
      auto point = [&](int i) { return i == TRI_THREADS - 1 ? top : top - w * exp2(-55.0 / TRI_THREADS * i); };
      const int n = below(sturm_minors(a, b2, k, point(t)) > 0);
      if (n > 0) lo = fmax(lo, point(n - 1));
      if (n < TRI_THREADS) hi = point(n);
    }
  }
  multisect<TRI_THREADS>(a, b2, k, 0, t, below, lo, hi);
  if (t >= 32) return;
  const double theta = 0.5 * (lo + hi);
  if (!twisted_vector(a, b, ib, k, theta, f, g, c1)) inverse_iteration(a, b, k, theta, scale, g, c1, f);
  if (t == 0) {
    out[0] = theta;
    out[1] = fabs(beta[k - 1]) * fabs(f[k - 1]);
  }
}

// The Ritz pair that an update ends with: s = unit eigenvector (s[0] >= 0),
// out[0] = its Rayleigh quotient, out[1] as above.  One warp, once per Lanczos
// run; the bracket and the vector do not depend on what the checks before it
// found (the vector becomes the node tensor, to the last place).
__global__ void __launch_bounds__(32) tridiag_vector_kernel(const double* __restrict__ alpha,
                                                            const double* __restrict__ beta, int k, double* out,
                                                            double* s) {
  __shared__ double a[TRI_MAX], b[TRI_MAX], b2[TRI_MAX], ib[TRI_MAX], x[TRI_MAX], cp[TRI_MAX], inv[TRI_MAX];
  const int t = threadIdx.x;
  double lo, hi, scale;
  stage_tridiag(alpha, beta, k, a, b, b2, ib, lo, hi, scale);
  multisect<32>(a, b2, k, 0, t, WarpBelow(), lo, hi);
  inverse_iteration(a, b, k, 0.5 * (lo + hi), scale, cp, inv, x);
  for (int i = t; i < k; i += 32) {
    double v = a[i] * x[i];
    if (i > 0) v += b[i - 1] * x[i - 1];
    if (i < k - 1) v += b[i] * x[i + 1];
    cp[i] = v;
    s[i] = x[i];
  }
  __syncwarp();
  const double rq = chain_dot(x, cp, k);
  if (t == 0) {
    out[0] = rq;
    out[1] = fabs(beta[k - 1]) * fabs(x[k - 1]);
  }
}

// Thick restart of a Lanczos cycle (Wu and Simon's thick-restart Lanczos).
// From the k x k tridiagonal T (alpha, beta; beta[k-1] couples the residual
// vector r) keep the m lowest Ritz pairs (theta_i, s_i).  Their couplings to
// r are c_i = beta[k-1] s_i[k-1].  A Lanczos process on diag(theta) started
// from c / |c| gives an orthogonal U (m x p) and a p x p tridiagonal; in
// reversed order the kept vectors Z = V S U form a tridiagonal block whose
// last vector alone couples to r with |c|, so the next cycle continues the
// ordinary three-term recurrence from r at position p.  Writes C = S U
// reversed (k x p, row-major: C[r * p + i]), alpha[0..p), beta[0..p) (beta[p-1]
// = |c|) and *p_out.
//
// One warp per Ritz pair: eigenvalues, factorisations and first solves side by
// side.  Vector i is kept orthogonal to the lower ones (twice per inverse
// iteration), so the vectors are finished one after another; its first pass
// over a lower vector runs beside the other warps' as soon as that one is
// final.  Bound by FP64 chains of k; 3.5 ms with everything in one lane.
__global__ void __launch_bounds__(32 * RESTART_MAX) lanczos_restart_kernel(double* alpha, double* beta, int k, int m,
                                                                           double* C, int* p_out) {
  __shared__ double a[TRI_MAX], b[TRI_MAX], b2[TRI_MAX], ib[TRI_MAX];
  __shared__ double S[RESTART_MAX][TRI_MAX], cp[RESTART_MAX][TRI_MAX], inv[RESTART_MAX][TRI_MAX];
  __shared__ double th[RESTART_MAX], U[RESTART_MAX][RESTART_MAX], w[RESTART_MAX], bracket[3];
  __shared__ int p_kept;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp == 0) {
    double glo, ghi, scale;
    stage_tridiag(alpha, beta, k, a, b, b2, ib, glo, ghi, scale);
    if (lane == 0) { bracket[0] = glo; bracket[1] = ghi; bracket[2] = scale; }
  }
  __syncthreads();
  const double scale = bracket[2];
  if (m > k) m = k;
  double* x = S[warp];
  if (warp < m) {
    double lo = bracket[0], hi = bracket[1];
    multisect<32>(a, b2, k, warp, lane, WarpBelow(), lo, hi);
    const double theta = 0.5 * (lo + hi);
    if (lane == 0) th[warp] = theta;
    inverse_lu(a, b, k, theta, scale, cp[warp], inv[warp]);
    inverse_start(x, k, warp);
    inverse_solve(b, k, cp[warp], inv[warp], x);
  }
  for (int done = 0; done < m; ++done) {
    if (warp == done) {
      for (int it = 0; it < INV_ITERS; ++it) {
        if (it > 0) inverse_solve(b, k, cp[warp], inv[warp], x);
        for (int pass = it > 0 ? 0 : 1; pass < 2; ++pass)
          for (int q = 0; q < warp; ++q) remove_along(S[q], x, k);
        make_unit(x, k);
      }
      if (warp == 0 && x[0] < 0.0)
        for (int i = lane; i < k; i += 32) x[i] = -x[i];
    }
    __syncthreads();
    if (warp > done && warp < m) remove_along(S[done], x, k);
  }
  __syncthreads();
  if (warp == 0) {
    // Lanczos on diag(theta) from c / |c| with full reorthogonalisation, one
    // kept pair per lane, sums in the order of the pairs
    const bool in = lane < m;
    const double t = in ? th[in ? lane : 0] : 0.0;
    const double c = in ? beta[k - 1] * S[in ? lane : 0][k - 1] : 0.0;
    auto put = [&](double v) {
      __syncwarp();
      if (in) w[lane] = v;
      __syncwarp();
    };
    auto dot = [&](const double* u) {   // u . w
      double h = 0.0;
      for (int i = 0; i < m; ++i) h = fma(u[i], w[i], h);
      return h;
    };
    put(c);
    const double cn = sqrt(dot(w));
    double la[RESTART_MAX], lb[RESTART_MAX];
    int p = 0;
    if (cn > 0.0) {
      if (in) U[0][lane] = c / cn;
      p = 1;
#pragma unroll
      for (int j = 0; j < RESTART_MAX; ++j) {
        if (j >= m || j >= p) break;
        __syncwarp();
        double v = in ? t * U[j][lane] : 0.0;
        put(v);
        la[j] = dot(U[j]);
        for (int pass = 0; pass < 2; ++pass)
          for (int q = 0; q <= j; ++q) {
            const double h = dot(U[q]);
            if (in) v = fma(-h, U[q][lane], v);
            put(v);
          }
        const double bj = sqrt(dot(w));
        if (j + 1 >= m || bj <= 1e-13 * fmax(scale, 1e-300)) break;
        if (j + 1 < RESTART_MAX) {
          lb[j] = bj;
          if (in) U[j + 1][lane] = v / bj;
        }
        p = j + 2;
      }
    }
    if (p == 0) {   // r decoupled: keep the lowest Ritz vector alone
      p = 1;
      if (in) U[0][lane] = lane == 0 ? 1.0 : 0.0;
      la[0] = th[0];
    }
    if (lane == 0) {   // reversed tridiagonal
#pragma unroll
      for (int i = 0; i < RESTART_MAX; ++i)
        if (i < p) {
          alpha[p - 1 - i] = la[i];
          if (i + 1 < p) beta[p - 2 - i] = lb[i];
        }
      beta[p - 1] = cn;
      *p_out = p_kept = p;
    }
  }
  __syncthreads();
  // C[:, i] = S^T U[p-1-i]
  const int p = p_kept;
  for (int e = threadIdx.x; e < k * p; e += blockDim.x) {
    const int r = e / p, i = e - r * p;
    double v = 0.0;
    for (int q = 0; q < m; ++q) v = fma(S[q][r], U[p - 1 - i][q], v);
    C[e] = v;
  }
}

// Z[:, i] = sum_r V[:, r] C[r * p + i] for i < p (p <= RESTART_MAX).
__global__ void rotate_basis_kernel(const double* __restrict__ V, long long ld, int k, const double* __restrict__ C,
                                    int p, double* __restrict__ Z, long long n) {
  __shared__ double cs[TRI_MAX * RESTART_MAX];
  for (int e = threadIdx.x; e < k * p; e += blockDim.x) cs[e] = C[e];
  __syncthreads();
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    double acc[RESTART_MAX];
#pragma unroll
    for (int q = 0; q < RESTART_MAX; ++q) acc[q] = 0.0;
    for (int r = 0; r < k; ++r) {
      const double v = V[(long long)r * ld + i];
#pragma unroll
      for (int q = 0; q < RESTART_MAX; ++q)
        if (q < p) acc[q] = fma(cs[r * p + q], v, acc[q]);
    }
#pragma unroll
    for (int q = 0; q < RESTART_MAX; ++q)
      if (q < p) Z[(long long)q * ld + i] = acc[q];
  }
}

int grid_for(long long n) {
  long long g = (n + 255) / 256;
  if (g > 152 * 8) g = 152 * 8;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

void launch_kc_gemm(const KTile* tiles, int n_tiles, const KOutput* outs, const KChunk* chunks, double* scratch,
                    cudaStream_t s, int fp32, int shape) {
  if (n_tiles <= 0) return;
#define QED_KC(T, BM, BN) kc_gemm_kernel<T, BM, BN><<<n_tiles, THREADS, 0, s>>>(tiles, outs, chunks, scratch)
#define QED_KC_ALL(T)                       \
  switch (shape) {                          \
    case KS_16: QED_KC(T, 16, 16); break;   \
    case KS_64: QED_KC(T, 64, 64); break;   \
    case KS_16x64: QED_KC(T, 16, 64); break; \
    case KS_64x16: QED_KC(T, 64, 16); break; \
    default: QED_KC(T, 32, 32); break;      \
  }
  if (fp32 == 1) {
    QED_KC_ALL(float)
  } else if (fp32 == 2) {
    QED_KC_ALL(ff)
  } else {
    QED_KC_ALL(double)
  }
#undef QED_KC_ALL
#undef QED_KC
  count_launches(1);
}

void launch_kc_reduce(const KOutput* outs, int n_outs, const int* red_list, int n_red, double* scratch,
                      cudaStream_t s) {
  if (n_red <= 0) return;
  dim3 grid(8, n_red);
  kc_reduce_kernel<<<grid, 256, 0, s>>>(outs, red_list, scratch);
  count_launches(1);
}

void launch_dot(const double* x, const double* y, long long n, double* partial, double* out, cudaStream_t s) {
  dot_partial_kernel<<<RED_BLOCKS, RED_THREADS, 0, s>>>(x, y, n, partial);
  count_launches(1);
  finish_kernel<<<1, RED_THREADS, 0, s>>>(partial, RED_BLOCKS, out);
  count_launches(1);
}

void launch_combine(const double* Q, long long ldq, int k, const double* c, double* x, long long n,
                    cudaStream_t s) {
  combine_kernel<<<grid_for(n), 256, 0, s>>>(Q, ldq, k, c, x, n);
  count_launches(1);
}

void launch_sqrt(const double* in, double* out, cudaStream_t s) {
  sqrt_kernel<<<1, 32, 0, s>>>(in, out);
  count_launches(1);
}

void launch_axpby(const double* x, double* y, long long n, const double* a_dev, double a_const, double a_sign,
                  const double* b_dev, double b_const, cudaStream_t s) {
  axpby_kernel<<<grid_for(n), 256, 0, s>>>(x, y, n, a_dev, a_const, a_sign, b_dev, b_const);
  count_launches(1);
}

void launch_scale_inv_sqrt(const double* x, double* y, long long n, const double* nrm2, cudaStream_t s,
                           const int* gate) {
  scale_inv_sqrt_kernel<<<grid_for(n), 256, 0, s>>>(x, y, n, nrm2, gate);
  count_launches(1);
}

void launch_copy(const double* x, double* y, long long n, cudaStream_t s) {
  copy_kernel<<<grid_for(n), 256, 0, s>>>(x, y, n);
  count_launches(1);
}

void launch_fill_uniform(double* x, long long n, uint64_t seed, uint64_t start, cudaStream_t s) {
  if (n <= 0) return;
  fill_uniform_kernel<<<grid_for(n), 256, 0, s>>>(x, n, seed, start);
  count_launches(1);
}

void launch_add_scaled(const double* x, double* y, long long n, double a, cudaStream_t s) {
  add_scaled_kernel<<<grid_for(n), 256, 0, s>>>(x, y, n, a);
  count_launches(1);
}

void launch_sum_rows(const double* x, long long n, int rows, double* y, cudaStream_t s) {
  sum_rows_kernel<<<grid_for(n), 256, 0, s>>>(x, n, rows, y);
  count_launches(1);
}

void launch_zero(double* x, long long n, cudaStream_t s) {
  if (n <= 0) return;
  zero_kernel<<<grid_for(n), 256, 0, s>>>(x, n);
  count_launches(1);
}

void launch_check_finite(const double* x, long long n, int* flag, cudaStream_t s) {
  if (n <= 0) return;
  check_finite_kernel<<<grid_for(n), 256, 0, s>>>(x, n, flag);
  count_launches(1);
}

void launch_to_float(const double* x, float* y, long long n, cudaStream_t s) {
  to_float_kernel<<<grid_for(n), 256, 0, s>>>(x, y, n);
  count_launches(1);
}

void launch_to_double(const float* x, double* y, long long n, cudaStream_t s) {
  to_double_kernel<<<grid_for(n), 256, 0, s>>>(x, y, n);
  count_launches(1);
}

void launch_cholesky_inv(double* G, double* Rinv, const long long* off, const int* n, const int* ld, int count,
                         int max_n, double ill_cond, int* status, cudaStream_t s) {
  if (count <= 0) return;
  allow_smem((const void*)cholesky_inv_kernel, 160 * 161 * 8);
  cholesky_inv_kernel<<<count, 256, (size_t)max_n * (max_n | 1) * sizeof(double), s>>>(G, Rinv, off, n, ld, status,
                                                                                  ill_cond);
  count_launches(1);
}

void launch_cgs2_qr(double* X, const long long* xoff, const int* rows, const int* cols, int count, double* R,
                    const long long* roff, int ldr, double dep_tol, double accept, cudaStream_t s) {
  if (count <= 0) return;
  cgs2_qr_kernel<<<count, QR_THREADS, 0, s>>>(X, xoff, rows, cols, R, roff, ldr, dep_tol, accept);
  count_launches(1);
}

void launch_lanczos_restart(double* alpha, double* beta, int k, int m, double* C, int* p_out, cudaStream_t st) {
  if (k <= 0 || k > TRI_MAX || m < 1 || m > RESTART_MAX) return;
  lanczos_restart_kernel<<<1, 32 * RESTART_MAX, 0, st>>>(alpha, beta, k, m, C, p_out);
  count_launches(1);
}

void launch_rotate_basis(const double* V, long long ld, int k, const double* C, int p, double* Z, long long n,
                         cudaStream_t st) {
  if (k <= 0 || k > TRI_MAX || p < 1 || p > RESTART_MAX) return;
  rotate_basis_kernel<<<grid_for(n), 256, 0, st>>>(V, ld, k, C, p, Z, n);
  count_launches(1);
}

void launch_tridiag_lowest(const double* alpha, const double* beta, int k, double* out, cudaStream_t st,
                           const double* prev) {
  if (k <= 0 || k > TRI_MAX) return;
  tridiag_lowest_kernel<<<1, TRI_THREADS, 0, st>>>(alpha, beta, k, out, prev);
  count_launches(1);
}

void launch_tridiag_vector(const double* alpha, const double* beta, int k, double* out, double* s, cudaStream_t st) {
  if (k <= 0 || k > TRI_MAX) return;
  tridiag_vector_kernel<<<1, 32, 0, st>>>(alpha, beta, k, out, s);
  count_launches(1);
}

}  // namespace qed
