// Device kernels of the TTN hot path (declarations shared by the engine).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace qed {

// Number of kernels launched by this library since load (all streams).
long long launch_count();
void count_launches(int n);
// Lets `kern` use up to `bytes` of dynamic shared memory on the current device:
// one attribute call per kernel and device (a call costs as much as a launch).
void allow_smem(const void* kern, int bytes);

// One contribution A(MxK) * B(KxN) to an output.  Element addressing:
//   A[m,k] = sA * aval[m] * A[row*a_m + k*a_k],  amap[m] = (row << 1) | negate, -1 = zero row
//   B[k,n] = sB * bval[k] * B[row*b_k + n*b_n],  bmap[k] likewise (maps and vals optional)
// With add != 0 there is no B:  C[m,n] += alpha * A[m,n] (A[m,n] addressed as A[m,k=n]).
// Two-level K (kin > 0): k stands for (k / kin, k % kin) and adds (k / kin) *
// a_ko + (k % kin) * a_k (b_ko, b_k in B), so that a contraction over two legs
// around a third is one chunk.  Two-level N (nin > 0 in the output) likewise,
// with b_no in B and c_no in C.  kdiv, ndiv: ceil(2^32 / kin), ceil(2^32 / nin).
struct KChunk {
  const double* A;
  long long a_m, a_k;
  const int* amap;
  const double* aval;
  const double* B;
  long long b_k, b_n;
  const int* bmap;
  const double* bval;
  int K;
  int add;
  double alpha;
  long long a_ko, b_ko, b_no;
  int kin;
  unsigned kdiv;
};

// An output C (MxN, C[m,n] at C + m*c_m + n*c_n) = sum of its chunks
// (accumulate != 0: C += sum).
struct KOutput {
  double* C;
  long long c_m, c_n;
  int M, N;
  int chunk_begin, chunk_end;
  int accumulate;
  int n_parts;        // > 1: split over chunk ranges, partial sums in scratch
  long long part_off; // scratch offset (doubles) of this output's partials
  long long c_no;
  int nin;
  unsigned ndiv;
};

// One CTA's work: a BM x BN tile of an output over a chunk range.
struct KTile {
  int out;
  int m0, n0;
  int chunk_begin, chunk_end;
  int part;           // partial slot (-1: write C directly)
};

constexpr int KT_BM = 32;   // tile of the default shape
constexpr int KT_BN = 32;
// Tile shapes of the grouped GEMM (rows x columns of the output tile):
// 16x16, 32x32, 64x64, and the flat 16x64 / 64x16 for outputs with few rows
// (leg operators applied to a node tensor) or few columns.
enum KcShape { KS_16 = 0, KS_32 = 1, KS_64 = 2, KS_16x64 = 3, KS_64x16 = 4, KS_COUNT = 5 };
inline int kc_shape_m(int shape) {
  static const int m[KS_COUNT] = {16, 32, 64, 16, 64};
  return m[shape];
}
inline int kc_shape_n(int shape) {
  static const int n[KS_COUNT] = {16, 32, 64, 64, 16};
  return n[shape];
}

// fp32 = 1: same contraction with FP32 multiply-accumulate (operands
// rounded to FP32 on load, results stored as FP64); fp32 = 2: float-float
// arithmetic on the FP32 pipes (operands split into two FP32 numbers, about
// 48 significant bits; FP64-level accuracy).  shape: the tile shape the
// tiles were cut with.
void launch_kc_gemm(const KTile* tiles, int n_tiles, const KOutput* outs, const KChunk* chunks,
                    double* scratch, cudaStream_t s, int fp32 = 0, int shape = KS_32);
void launch_kc_reduce(const KOutput* outs, int n_outs, const int* red_list, int n_red, double* scratch,
                      cudaStream_t s);

// ---- bottom-node products as packed row gathers (kernels_bh.cu) ----
// Output sector of y (M x N, row-major): the sum over its chunks of
//   K > 0:  alpha s(r) val(r) A[map(r) * ld + k] B[k, n]  (alpha B staged at w)
//   K = 0:  alpha s(r) val(r) A[map(r) * ld + n]
// with map sign-encoded as in KChunk (NULL: identity) and val optional.
// div: ceil(2^32 / K) or, in an output, ceil(2^32 / N).
struct BhChunk {
  const double* A;
  const int* map;
  const double* val;
  long long w;
  double alpha;
  int ld, K;
  unsigned div;
};
struct BhOut {
  double* C;
  int M, N;
  int chunk_begin, chunk_end;
  unsigned div;
};
struct BhTile {
  int out;
  int row0;
};
// Staging job: w[off + k * N + n] = alpha B[k * b_k + n * b_n].
struct BhJob {
  const double* B;
  long long b_k, b_n;
  long long off;
  double alpha;
  int K, N;
};
// Rows of a tile for outputs up to max_n and terms up to max_k wide (at most 160:
// the widest sector that the QR of a centre move takes).
int bh_rows(int max_n, int max_k);
// w: staging of 8 bytes per entry.  ff_arith: float-float arithmetic.
void launch_bh(const BhTile* tiles, int n_tiles, const BhOut* outs, const BhChunk* chunks, const BhJob* jobs,
               int n_jobs, int max_n, int max_k, double* w, cudaStream_t s, int ff_arith);

// ---- vector kernels (FP64) ----
// partial sums per block then a single-block finish: deterministic.
void launch_dot(const double* x, const double* y, long long n, double* partial, double* out, cudaStream_t s);
// x = sum_j c[j] Q_j
void launch_combine(const double* Q, long long ldq, int k, const double* c, double* x, long long n, cudaStream_t s);
// One Lanczos step after y = H v_{k-1} (kernels_lz.cu; V holds v_0 .. v_{k-1},
// columns of stride ldq, k <= 128): alpha_j = v_j . y, the three-term residual
// w' = y - alpha_j v_j - beta_{j-1} v_{j-1} (beta_prev, unused for k = 1),
// classical Gram-Schmidt of w' against all k vectors, a second pass when the
// first left less than ratio |w'|^2 (Daniel-Gragg-Kaufman-Stewart, decided on
// the device), then beta_j = |w| and v_next = w / |w|.  y is overwritten.
// partial: kLzPartial doubles; coef: 256 doubles; bar: two zeroed counters,
// zero again afterwards.  polls: bound of each grid barrier's wait (< 0: the
// default, 2^22); a wait that runs out sets *err, and a step that finds *err set
// does nothing: both leave alpha_j = beta_j = 0, which ends the run.  ff_arith
// != 0: dots and updates in float-float arithmetic (the data stay FP64).
struct LzStep {
  const double* V;
  long long ldq;
  int k;
  double* y;
  long long n;
  double* partial;
  double* coef;
  double ratio;
  double* alpha_j;
  const double* beta_prev;
  double* beta_j;
  double* v_next;
  unsigned* bar;
  int* err;
  long long polls;
};
constexpr int kLzRowBlocks = 1216;   // a sum's row blocks: its order does not depend on the grid
constexpr long long kLzPartial = 132LL * kLzRowBlocks;
int launch_lz_step(const LzStep& p, int ff_arith, cudaStream_t s);
// out[0] = sqrt(max(in[0], 0))
void launch_sqrt(const double* in, double* out, cudaStream_t s);
// y = a*x + b*y with a, b read from device scalars (nullable -> constants)
void launch_axpby(const double* x, double* y, long long n, const double* a_dev, double a_const, double a_sign,
                  const double* b_dev, double b_const, cudaStream_t s);
// y = x / sqrt(*nrm2) ; returns nothing
// (nothing is written where *gate, if given, is not zero)
void launch_scale_inv_sqrt(const double* x, double* y, long long n, const double* nrm2, cudaStream_t s,
                           const int* gate = nullptr);
void launch_copy(const double* x, double* y, long long n, cudaStream_t s);
void launch_fill_uniform(double* x, long long n, uint64_t seed, uint64_t start, cudaStream_t s);
void launch_add_scaled(const double* x, double* y, long long n, double a, cudaStream_t s);
// y[i] = sum over r < rows of x[r * n + i]
void launch_sum_rows(const double* x, long long n, int rows, double* y, cudaStream_t s);
void launch_zero(double* x, long long n, cudaStream_t s);
void launch_to_float(const double* x, float* y, long long n, cudaStream_t s);
// *flag = 1 if any of x[0..n) is NaN or infinite (flag untouched otherwise).
void launch_check_finite(const double* x, long long n, int* flag, cudaStream_t s);
void launch_to_double(const float* x, double* y, long long n, cudaStream_t s);

// ---- small dense linear algebra (one CTA per matrix) ----
// For each matrix i: G_i (n_i x n_i at G + off_i, leading dim ld_i): in-place
// upper Cholesky R (G = R^T R) and then Rinv = R^{-1} (written to Rinv + off_i).
// status[i] = 0 ok, 1 non-positive pivot.
// status[i] = 2 when a pivot R_jj^2 <= ill_cond * max_j G_jj (ill-conditioned).
// max_n: largest n over the batch (<= 160).
void launch_cholesky_inv(double* G, double* Rinv, const long long* off, const int* n, const int* ld, int count,
                         int max_n, double ill_cond, int* status, cudaStream_t s);
// Gram-Schmidt QR (two passes per column) with deterministic completion of
// dependent columns; one CTA per column-major sector matrix (n <= 256).
void launch_cgs2_qr(double* X, const long long* xoff, const int* rows, const int* cols, int count, double* R,
                    const long long* roff, int ldr, double dep_tol, double accept, cudaStream_t s);

// Lowest eigenvalue of the symmetric tridiagonal (alpha[0..k), beta[0..k-1))
// (1 <= k <= 128).  out[0] = theta, out[1] = |beta[k-1] * s_k| (Ritz residual
// estimate; beta[k-1] is the trailing coupling).  prev (optional, device): an
// upper bound of theta, e.g. the value for a smaller basis of the same run; a
// wrong one costs a round, not the result.
void launch_tridiag_lowest(const double* alpha, const double* beta, int k, double* out, cudaStream_t s,
                           const double* prev = nullptr);
// The same with the unit eigenvector in svec[0..k) (svec[0] >= 0) and its
// Rayleigh quotient in out[0].
void launch_tridiag_vector(const double* alpha, const double* beta, int k, double* out, double* svec, cudaStream_t s);
// Thick restart (keep the m <= 8 lowest Ritz pairs of the k x k tridiagonal,
// k <= 128): writes the k x p combination C (row-major), the new leading
// p x p tridiagonal into alpha/beta with beta[p-1] the coupling to the
// residual vector, and p (1 <= p <= m) to *p_out.
void launch_lanczos_restart(double* alpha, double* beta, int k, int m, double* C, int* p_out, cudaStream_t s);
// Z[:, i] = sum_r V[:, r] C[r * p + i], i < p <= 8 (columns of length n, stride ld).
void launch_rotate_basis(const double* V, long long ld, int k, const double* C, int p, double* Z, long long n,
                         cudaStream_t s);

}  // namespace qed

namespace qed {

// ---- mixed-precision bottom-node H_eff (tcgen05) ----
// One output c-sector of y (rows x n, FP64, row-major with ld = n) is the
// sum of GEMM chunks  sign(r) * X[map(r), :] . W^T  accumulated in TMEM
// (A rows gathered into shared memory, B = W, both K-major) and of add terms
// alpha * sign(r) * val(r) * X32[map(r), :n], added in FP64 when the tile is
// written; X32 and ld are the same in all adds of an output.
struct TcChunk {
  const void* X;      // staging source sector matrix (BF16 or FP32), row stride xstride
  const int* map;     // sign-encoded row map (nullable: identity)
  const void* W;      // B operand in core-matrix order (alpha folded in; split: [hi | lo])
  int kpad;           // K of the staged rows, multiple of 16 (split: of each part)
  int xstride;        // elements per staged source row
};
struct TcAdd {
  const float* X32;   // FP32 staging source sector matrix, row stride ld
  const int* map;     // nullable: identity
  const double* val;  // nullable
  double alpha;
  int ld;
};
struct TcOutput {
  double* y;
  const int* order;   // row of the sector that row i of the tiles' order is
  int rows, n, npad;
  int add_begin, add_end;
  unsigned div;       // ceil(2^32 / n)
};
// 128 rows of an output, and the chunks that reach one of them.
struct TcTile {
  int out;
  int row0;
  int chunk_begin, chunk_end;
};
// Staging of x: dst32 (and, for BF16 and split operands, dst), rows x kpad, zero
// padded, <- src (rows x cols, ld_src), FP64 source.
struct ConvJob {
  const double* src;
  long long ld_src;   // row stride of the source
  void* dst;          // BF16 rows, or split rows [hi | lo] of 2 kpad floats
  float* dst32;       // FP32 copy
  int rows, cols, kpad;
};
// Staging of one environment block: dst (npad x kpad, core-matrix order) <-
// scale * src (rows x cols, ld_src).
struct WJob {
  const double* src;
  long long ld_src;
  void* dst;
  int rows, cols, npad, kpad;
  double scale;
};

// elem: 2 = BF16 operands (kind::f16), 4 = TF32 operands (kind::tf32).
// split (TF32 only): both operands as hi + lo TF32 parts; three sub-products
// x_hi W_hi + x_hi W_lo + x_lo W_hi whose sum carries about 21 bits (x_lo W_lo
// dropped).  y_shift: added to every output pointer (elements), so that one
// plan serves any y.
// err: device flag set to 1 if a wait timed out (results then invalid).
// polls: bound of each mbarrier wait in polls (< 0: the default, 2^22).
int launch_tc_heff(int elem, int split, const TcTile* tiles, int n_tiles, const TcOutput* outs,
                   const TcChunk* chunks, const TcAdd* adds, int max_kpad, int max_npad, long long y_shift, int* err,
                   cudaStream_t s, long long polls = -1);
// ---- grouped leg contractions on the tensor cores (tcgen05) ----
// One contribution D[r, j] += alpha * sum_{k < K} A(r, k) B(j, k):
//   A(r, k) = A[(r / R2) * s1 + (r % R2) * s2 + k * sk]  (float if a_f32, else double)
//   B(j, k) = B[j * bj + k * bk]                          (double)
struct TgChunk {
  const void* A;
  long long s1, s2, sk;
  const double* B;
  long long bj, bk;
  int R2;
  int K;
  int a_f32;
  float alpha;
  unsigned r2div;   // ceil(2^32 / R2); 0: every row below R2
};
// An output: D[r, j] (r < rows, j < N) at C[(r / R2) * t1 + (r % R2) * t2 + j * cj],
// float if c_f32 (else double), written or added (accumulate); chunks of its
// tiles are summed in one accumulator; n_parts > 1: tiles write FP32 partial
// sums (rows x N each, at scratch + part_off) that the reduction adds up.
struct TgOut {
  void* C;
  long long t1, t2, cj;
  int R2;
  int rows, N, npad;
  int c_f32;
  int accumulate;
  int n_parts;
  long long part_off;
  unsigned r2div;   // as in TgChunk
};
// One CTA: rows row0 .. row0 + 127 of output `out` over chunks [chunk_begin,
// chunk_end); part >= 0 writes partial slot `part`.  n_sub > 0: a group of
// outputs out .. out + n_sub - 1, output out + i from the one chunk chunk_begin
// + i, with the same rows, K, padded width and A operand in all of them.
struct TgTile {
  int out;
  int row0;
  int chunk_begin, chunk_end;
  int part;
  int n_sub;
};
constexpr int kTgGroup = 64;   // most columns of a group
// Shared memory of one launch (two stages of A and B tiles).
int tg_stage_bytes(int elem, int split, int max_npad, int* a_bytes, int* b_bytes);
// elem 4: TF32 operands (split: three products of hi / lo parts), 2: BF16.
// max_npad: widest tile (a group's columns together).  red_list: outputs with
// n_parts > 1 (reduced after the GEMM).  x_shift, y_shift: added to every FP64
// A and C pointer (elements), so that one plan serves any x and y.  err: device
// flag set if a wait timed out; polls < 0: default bound.
int launch_tg_gemm(int elem, int split, const TgTile* tiles, int n_tiles, const TgOut* outs, const TgChunk* chunks,
                   int max_npad, float* scratch, const int* red_list, int n_red, long long x_shift, long long y_shift,
                   int* err, cudaStream_t s, long long polls = -1);

// ---- FP64-accurate contractions on the BF16 tensor cores (digit planes) ----
constexpr int kOzDigits = 5;   // balanced base-256 digits per FP64 entry (about 2^-39 of the max)
// planes (16 bytes per entry, 8 BF16 planes of which kOzDigits are used)
// <- x[0..n), relative to 2^E >= max |x| (max |x| written to *amax).
void launch_oz_slice(const double* x, long long n, double* amax, void* planes, cudaStream_t s);
// Job: for one term and output sector, rows (c < cols) of the source sector
// matrix (at a_off, row stride a_ld, in planes) selected by map (sign-encoded
// source row per output row; NULL = identity).  Its FP64 partial blocks
// [part][c][c'] start at part_off.
struct OzJob {
  const int* map;
  long long a_off;
  long long part_off;
  int a_ld;
  int cols;
};
// CTA: jobs [job_begin, job_end) stacked in slots of `slot` MMA rows, against
// output sector rows [r0, r1) (at b_off, row stride b_ld, n columns c'),
// writing partial slot `part` of each job.
struct OzTile {
  long long b_off;
  int b_ld, n;
  int r0, r1;
  int job_begin, job_end;
  int slot;
  int part;
};
// One operator block O[c', c] (ld) += sum over its entries of alpha * the
// sum of that job's partial blocks.
struct OzSum {
  long long off;          // job's part_off
  long long part_stride;  // cols * n
  int n_parts;
  double alpha;
};
struct OzOut {
  double* O;
  int ld;
  int rows, cols;         // c' (output sector) x c (source sector)
  int sum_begin, sum_end;
};
// npad: MMA width (32 or 64, >= every tile's n).  err: set if a wait timed out.
int launch_oz_gram(const OzTile* tiles, int n_tiles, const OzJob* jobs, const void* planes, int npad, double* partial,
                   const OzOut* outs, int n_outs, const OzSum* sums, int* err, cudaStream_t s, long long polls = -1);

// Staging for launch_tc_heff; shift: added to every source pointer (elements).
void launch_convert(int elem, int split, const ConvJob* jobs, int n_jobs, long long max_elems, long long shift,
                    cudaStream_t s);
void launch_stage_w(int elem, int split, const WJob* jobs, int n_jobs, cudaStream_t s);

}  // namespace qed
