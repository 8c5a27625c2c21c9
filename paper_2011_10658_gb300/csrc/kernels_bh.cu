// Bottom-node H_eff x in FP64 and float-float arithmetic.
//
// y[r, :] = sum_c alpha_c s_c(r) X_c[map_c(r), :] B_c  +  sum_a alpha_a s_a(r) X_a[map_a(r), :]
//
// A site operator keeps one source row per output row or none (Eq. (15), the
// plaquette factors and the projectors of Eq. (16)), and most rows have none:
// at a corner pair of 4x4x4 a term selects a third of the rows on average.
// GB300 retires about two FP64 multiply-adds per clock and SM, so a dense
// tile over all rows and a padded column count (kc_gemm_kernel) spends most
// of that on zeros.  Here one warp owns 32 rows of one output sector and
// walks the terms: the lanes read the rows' map entries, the rows that have a
// source are packed (ballot), their source rows staged in shared memory in
// the arithmetic's own format, and the lanes run over (packed row, column)
// pairs, so that every multiply-add issued is one the term asks for.  Sums
// stay in shared memory until the last term; y is written once.  The
// environment blocks come transposed and scaled (bh_stage_kernel), so that
// the lanes read them along the columns.  Warps need no barrier of their
// CTA; the next term's map is read while the current one is worked on.
//
// Tiles (bh_rows): sectors that sum past 24 columns (output + term) take 16
// rows a warp, which leaves six warps per scheduler beside the sums and
// the staged rows; with 32 rows three fit and the FP64 pipe idled half the
// time.  Narrow sectors have too little work per term to hide its loads: there
// the four warps of a CTA share a 32-row tile and divide the terms.
//
// Bound by the FP64 pipe (four warps saturate it: 1.00 TFLOP/s measured).
// Whole products, GB300: bottom node 0 of 4x4x4 chi=64 3184 -> 1362 us (93 %
// of the pipe's cycles; 2200 us with 32-row tiles), 2x2x2 chi=8 1001 -> 51 us
// (62 us without the shared tiles), the eight products of an energy gradient
// at 4x4x4 chi=32 4590 -> 1610 us.
#include <algorithm>

#include "ffloat.cuh"
#include "kernels.cuh"

namespace qed {

namespace {

constexpr int BH_WARPS = 4;       // warps of a CTA
constexpr int BH_SMEM = 200 * 1024;

// e / d for the small item indices here (e d < 2^32): m = ceil(2^32 / d)
__device__ __forceinline__ int bh_div(int e, int d, unsigned m) { return d == 1 ? e : (int)__umulhi((unsigned)e, m); }

template <typename T>
__device__ __forceinline__ T bh_ld(const T* p);
template <>
__device__ __forceinline__ double bh_ld<double>(const double* p) { return __ldg(p); }
template <>
__device__ __forceinline__ ff bh_ld<ff>(const ff* p) {
  const float2 v = __ldg((const float2*)p);
  return ff(v.x, v.y);
}

// Environment blocks of one plan: dst[k * N + n] = alpha B[k, n].
template <typename T>
__global__ void bh_stage_kernel(const BhJob* __restrict__ jobs, T* __restrict__ dst) {
  const BhJob j = jobs[blockIdx.x];
  const T alpha = to_t<T>(j.alpha);
  for (int e = threadIdx.x; e < j.K * j.N; e += blockDim.x) {
    const int k = e / j.N, n = e - k * j.N;
    dst[j.off + e] = alpha * to_t<T>(j.B[(long long)k * j.b_k + (long long)n * j.b_n]);
  }
}

__device__ __forceinline__ double bh_neg(double v, int flip) {
  return __hiloint2double(__double2hiint(v) ^ (flip << 31), __double2loint(v));
}
__device__ __forceinline__ ff bh_neg(ff v, int flip) {
  const unsigned m = (unsigned)flip << 31;
  return ff(__uint_as_float(__float_as_uint(v.hi) ^ m), __uint_as_float(__float_as_uint(v.lo) ^ m));
}

// ROWS: rows of a warp's tile.  A lane works on two (packed row, column)
// pairs at a time while two are left.  SHARE: the warps of a CTA share one
// tile, each walks every BH_WARPS-th term, and their sums are added at the end.
template <typename T, int ROWS, bool SHARE>
__global__ void __launch_bounds__(32 * BH_WARPS) bh_kernel(const BhTile* __restrict__ tiles, int n_tiles,
                                                           const BhOut* __restrict__ outs,
                                                           const BhChunk* __restrict__ chunks,
                                                           const T* __restrict__ w, int max_n, int ldx) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ti = SHARE ? blockIdx.x : blockIdx.x * (blockDim.x >> 5) + warp;
  if (ti >= n_tiles) return;
  const int step = SHARE ? BH_WARPS : 1;
  const BhTile tile = tiles[ti];
  const BhOut out = outs[tile.out];
  const int N = out.N, rows = min(ROWS, out.M - tile.row0);
  const unsigned mn = out.div;
  const size_t per = (size_t)ROWS * ((max_n + ldx + 1) * sizeof(T) + 2 * sizeof(int));
  uint8_t* base = smem + (size_t)warp * per;
  T* acc = (T*)base;
  T* xs = acc + (size_t)ROWS * max_n;
  T* fac = xs + (size_t)ROWS * ldx;   // factor of a packed row in a term without environment operator
  int* row_of = (int*)(fac + ROWS);
  int* src_of = row_of + ROWS;
  for (int e = lane; e < rows * N; e += 32) acc[e] = T(0);
  const int r = tile.row0 + lane;
  auto map_entry = [&](int ci) {
    const int* map = chunks[ci].map;
    return lane < rows ? (map ? __ldg(map + r) : (r << 1)) : -1;
  };
  const int first = out.chunk_begin + (SHARE ? warp : 0);
  int next = first < out.chunk_end ? map_entry(first) : -1;
  __syncwarp();
  for (int ci = first; ci < out.chunk_end; ci += step) {
    const int src = next;
    if (ci + step < out.chunk_end) next = map_entry(ci + step);
    const unsigned live = __ballot_sync(0xffffffffu, src >= 0);
    if (!live) continue;
    const BhChunk c = chunks[ci];
    const int n_act = __popc(live);
    if (src >= 0) {
      const int p = __popc(live & ((1u << lane) - 1u));
      row_of[p] = lane;
      src_of[p] = src;
      T f = T(1);
      if (c.val) f = to_t<T>(__ldg(c.val + r));
      if (c.K == 0) f = f * to_t<T>(c.alpha);
      fac[p] = bh_neg(f, src & 1);
    }
    __syncwarp();
    if (c.K == 0) {
      // no environment operator: y[r, :] += alpha val(r) x[src, :]
      for (int e = lane; e < n_act * N; e += 32) {
        const int i = bh_div(e, N, mn), n = e - i * N;
        T* to = acc + row_of[i] * N + n;
        *to = kc_fma(fac[i], to_t<T>(__ldg(c.A + (long long)(src_of[i] >> 1) * c.ld + n)), *to);
      }
      __syncwarp();
      continue;
    }
    const int K = c.K;
#pragma unroll 2
    for (int e = lane; e < n_act * K; e += 32) {
      const int i = bh_div(e, K, c.div), k = e - i * K;
      const int s = src_of[i];
      T v = bh_neg(to_t<T>(__ldg(c.A + (long long)(s >> 1) * c.ld + k)), s & 1);
      if (c.val) v = bh_neg(v, s & 1) * fac[i];
      xs[i * ldx + k] = v;
    }
    __syncwarp();
    const T* wb = w + c.w;
    const int tot = n_act * N;
    for (int e0 = 0; e0 < tot; e0 += 64) {
      const int ea = min(e0 + lane, tot - 1), ia = bh_div(ea, N, mn), na = ea - ia * N;
      const T* xa = xs + ia * ldx;
      const T* wa = wb + na;
      T* ta = acc + row_of[ia] * N + na;
      T a = *ta;
      if (e0 + 32 < tot) {
        const int eb = min(e0 + 32 + lane, tot - 1), ib = bh_div(eb, N, mn), nb = eb - ib * N;
        const T* xb = xs + ib * ldx;
        const T* wbb = wb + nb;
        T* tb = acc + row_of[ib] * N + nb;
        T b = *tb;
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
          a = kc_fma(xa[k], bh_ld<T>(wa + k * N), a);
          b = kc_fma(xb[k], bh_ld<T>(wbb + k * N), b);
        }
        __syncwarp();
        if (e0 + 32 + lane < tot) *tb = b;
      } else {
#pragma unroll 8
        for (int k = 0; k < K; ++k) a = kc_fma(xa[k], bh_ld<T>(wa + k * N), a);
        __syncwarp();
      }
      if (e0 + lane < tot) *ta = a;
    }
    __syncwarp();
  }
  double* y = out.C + (long long)tile.row0 * N;
  if (SHARE) {
    __syncthreads();
    for (int e = threadIdx.x; e < rows * N; e += 32 * BH_WARPS) {
      T v = ((const T*)smem)[e];
#pragma unroll
      for (int u = 1; u < BH_WARPS; ++u) v = v + ((const T*)(smem + u * per))[e];
      y[e] = to_d<T>(v);
    }
    return;
  }
  for (int e = lane; e < rows * N; e += 32) y[e] = to_d<T>(acc[e]);
}

// Shared memory of a warp: 16 rows of 160 columns take 41 KB, four warps 165 of
// the SM's 227.  The rows of an odd leading dimension start in different banks.
size_t bh_warp_bytes(int max_n, int max_k, int rows) {
  return (size_t)rows * ((max_n + (max_k | 1) + 1) * 8 + 2 * sizeof(int));
}

template <typename T, int ROWS, bool SHARE>
void launch(const BhTile* tiles, int n_tiles, const BhOut* outs, const BhChunk* chunks, int max_n, int max_k,
            const double* w, cudaStream_t s) {
  const size_t per = bh_warp_bytes(max_n, max_k, ROWS);
  allow_smem((const void*)bh_kernel<T, ROWS, SHARE>, BH_SMEM);
  const int grid = SHARE ? n_tiles : (n_tiles + BH_WARPS - 1) / BH_WARPS;
  bh_kernel<T, ROWS, SHARE><<<grid, 32 * BH_WARPS, BH_WARPS * per, s>>>(tiles, n_tiles, outs, chunks, (const T*)w, max_n,
                                                                  max_k | 1);
  count_launches(1);
}

}  // namespace

int bh_rows(int max_n, int max_k) {
  return max_n + max_k > 24 ? 16 : 32;
}

void launch_bh(const BhTile* tiles, int n_tiles, const BhOut* outs, const BhChunk* chunks, const BhJob* jobs,
               int n_jobs, int max_n, int max_k, double* w, cudaStream_t s, int ff_arith) {
  if (n_tiles <= 0) return;
  if (n_jobs > 0) {
    if (ff_arith)
      bh_stage_kernel<ff><<<n_jobs, 256, 0, s>>>(jobs, (ff*)w);
    else
      bh_stage_kernel<double><<<n_jobs, 256, 0, s>>>(jobs, w);
    count_launches(1);
  }
  const bool wide = bh_rows(max_n, max_k) == 16;
  if (ff_arith)
    (wide ? launch<ff, 16, false> : launch<ff, 32, true>)(tiles, n_tiles, outs, chunks, max_n, max_k, w, s);
  else
    (wide ? launch<double, 16, false> : launch<double, 32, true>)(tiles, n_tiles, outs, chunks, max_n, max_k, w, s);
}

}  // namespace qed
