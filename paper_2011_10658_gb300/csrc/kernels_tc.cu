// Mixed-precision H_eff x for bottom TTN nodes on the sm_103a tensor cores.
//
// y[r, :] = sum_chunks s_c(r) X[map_c(r), :] W_c^T  +  sum_adds alpha val(r) X[map(r), :]
//
// The physical legs of a bottom node carry monomial site operators
// (Eq. (15) and the plaquette factors: at most one +-1 per row), so each
// product term becomes a row gather of the node tensor followed by one
// dense contraction with the environment operator on the parent leg.  The
// gather feeds the A operand of tcgen05.mma (no-swizzle K-major core matrices
// of 8 rows x 16 bytes), the environment block is the B operand, and all
// product terms of an output tile accumulate in one TMEM accumulator.  Terms
// without an environment factor (the diagonal of the two sites, the internal
// hopping) are added in FP64 when the tile is written.
//
// One CTA = one 128-row tile of one output charge sector.  The rows of a
// sector are ordered by the terms that reach them, so a tile walks only some
// of the terms (Engine::tc_tiles).  Eight gather warps feed two stages of A,
// one thread of a ninth warp copies the blocks of W (staged in core-matrix
// order, bulk copies two terms ahead) and issues the MMAs; they meet on
// mbarriers only.  x is staged once per product as FP32 rows, for the terms
// without environment factor, and as operand rows: BF16, or the hi and lo TF32
// parts of every entry (lo is what the FP64 entry leaves after hi: cutting both
// from the FP32 row would gather half as much, 22 us less per product of 4x4x4
// chi=64, but drops the bits that FP32 has rounded away).  A warp's load takes 8
// rows x 64 bytes: eight cache lines instead of one per lane, and stores that
// fill all banks.  The rows of term j + 1 and the map of term j + 2 are read
// while term j waits for its stage; rows two terms ahead in registers measured
// the same.
//
// Bound by the round trip gather -> MMA -> free stage of each term (two CTAs
// an SM for split TF32).  Product at bottom node 0 of 4x4x4, whole call, GB300:
// chi=64 split TF32 287 -> 139 us, chi=48 BF16 132 -> 87 us: coalesced gathers,
// gather and issue on separate warps, 16-byte pieces at compile-time places (a
// launch whose rows are narrow has a kernel with fewer registers: 159 us with
// one for all widths), rows ordered by their terms.  About 10 us are the FP64
// multiply-adds at the end, which float-float arithmetic on the FP32 pipes would
// save with fewer bits.
//
// Every mbarrier wait is bounded (polls, a launch argument); a timeout sets
// *err, and the CTA then drains its MMAs through a commit to a fresh barrier
// and its bulk copies through their own barriers (waited on with the default
// bound, so that nothing is in flight when TMEM is freed), and returns.
#include <algorithm>
#include <cuda_bf16.h>

#include <cstdio>
#include <type_traits>

#include "ffloat.cuh"
#include "kernels.cuh"

namespace qed {

namespace {

constexpr int TC_GATHER_WARPS = 8;
constexpr int TC_THREADS = 32 * (TC_GATHER_WARPS + 1);   // and the warp that issues copies and MMAs
constexpr int TC_WARP_ROWS = 16;                  // rows of A a warp gathers
constexpr int TC_ADDS = 8;                        // terms without environment factor whose row factors are held
constexpr int TC_UNROLL = 4;                      // outputs a thread writes at a time
constexpr long long kWaitPolls = 1LL << 22;   // default bound of one mbarrier wait

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: start address, leading-dimension byte
// offset (K-direction core-matrix stride), stride-dimension byte offset
// (8-row group stride), descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// byte offset of 16-byte chunk q of row r in a K-major no-swizzle tile
__device__ __forceinline__ uint32_t core_off(int r, int q, int kchunks) {
  return (uint32_t)(((r >> 3) * kchunks + q) * 128 + (r & 7) * 16);
}

__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity, long long polls = kWaitPolls) {
  for (long long it = 0; it < polls; ++it) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
    if (it > 32) __nanosleep(32);
  }
  return false;
}

__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar));
}

template <int ELEM>
__device__ __forceinline__ void mma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
  if (ELEM == 4)
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
  else
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ float tf32_hi(float x) { return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u); }

// One thread's share of a chunk's A tile: KQ / 2 pieces of 16 bytes, of a split
// row KQ / 2 of each part.  Piece `it` is piece q of row r of the warp's 16
// rows, the eight rows of a core matrix on neighbouring lanes.  mp: lane l holds
// the map entry of row l (mod 16).
template <int KQ, bool SPLIT>
struct Gather {
  static constexpr int PARTS = SPLIT ? 2 : 1, HALF = KQ / 2, N = HALF * PARTS;
  static __device__ __forceinline__ int group(int it, int lane) { return it * 4 + (lane >> 3) >= KQ ? 1 : 0; }
  static __device__ __forceinline__ int piece(int it, int lane) { return it * 4 + (lane >> 3) - group(it, lane) * KQ; }
  template <int ELEM>
  static __device__ __forceinline__ void load(uint4* v, const void* X, int row_bytes, int mp, int lane) {
    const int s0 = __shfl_sync(0xffffffffu, mp, lane & 7), s1 = __shfl_sync(0xffffffffu, mp, 8 + (lane & 7));
    const uint8_t* x0 = (const uint8_t*)X + (long long)(s0 >> 1) * row_bytes;
    const uint8_t* x1 = (const uint8_t*)X + (long long)(s1 >> 1) * row_bytes;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int it = i % HALF, part = i / HALF;
      const bool g = group(it, lane);
      v[i] = make_uint4(0u, 0u, 0u, 0u);
      if ((g ? s1 : s0) >= 0) v[i] = __ldg((const uint4*)((g ? x1 : x0) + (part * KQ + piece(it, lane)) * 16));
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int s = group(i % HALF, lane) ? s1 : s0;
      const uint32_t flip = s < 0 ? 0u : (ELEM == 2 ? (uint32_t)(s & 1) * 0x80008000u : (uint32_t)s << 31);
      v[i].x ^= flip; v[i].y ^= flip; v[i].z ^= flip; v[i].w ^= flip;
    }
  }
  static __device__ __forceinline__ void store(uint8_t* A, const uint4* v, int warp, int lane) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int it = i % HALF, part = i / HALF;
      *(uint4*)(A + ((warp * 2 + group(it, lane)) * PARTS * KQ + part * KQ + piece(it, lane)) * 128 + (lane & 7) * 16) = v[i];
    }
  }
};

// Row widths in pieces (of a part): a K step is 32 bytes, two pieces; 16 columns
// are two pieces of BF16, four of TF32.  f(integral_constant) of the width.
template <int KQ, int STEP, int MAXKQ, typename F>
__device__ __forceinline__ void by_width(int kq, F f) {
  if constexpr (KQ <= MAXKQ) {
    if (kq == KQ)
      f(std::integral_constant<int, KQ>());
    else
      by_width<KQ + STEP, STEP, MAXKQ>(kq, f);
  }
}

// A launch whose rows are at most NARROW pieces wide keeps two (split) or three
// CTAs on an SM; up to WIDE, what the stages of the widest rows leave in shared
// memory (see launch_tc_heff) is one or two.
template <int ELEM, bool SPLIT>
struct Width {
  static constexpr int STEP = ELEM, NARROW = SPLIT ? 8 : 12, WIDE = SPLIT ? 16 : (ELEM == 2 ? 20 : 24);
};

template <int ELEM, bool SPLIT, int MAXKQ>
__global__ void __launch_bounds__(TC_THREADS, (SPLIT ? 1 : 2) + (MAXKQ <= Width<ELEM, SPLIT>::NARROW ? 1 : 0))
    tc_heff_kernel(const TcTile* __restrict__ tiles, const TcOutput* __restrict__ outs,
                   const TcChunk* __restrict__ chunks, const TcAdd* __restrict__ adds, int a_bytes, int b_bytes,
                   int b_stages, long long y_shift, int* err, long long polls) {
  constexpr int PARTS = SPLIT ? 2 : 1, STEP = Width<ELEM, SPLIT>::STEP;
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ uint32_t tmem_slot;
  // MMAs of the two A stages, drain, the gathers of the two A stages, the
  // copies of up to four B stages
  __shared__ __align__(8) uint64_t mbar[9];
  __shared__ int s_fail;
  const TcTile tile = tiles[blockIdx.x];
  const TcOutput out = outs[tile.out];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint8_t* const B0 = smem + 2 * a_bytes;
  uint32_t ncols = 32;
  while ((int)ncols < out.npad) ncols <<= 1;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < 9; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&mbar[i])), "r"(i == 3 || i == 4 ? TC_GATHER_WARPS : 1));
    asm volatile("fence.mbarrier_init.release.cluster;");
    s_fail = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_slot;
  const int nchunks = tile.chunk_end - tile.chunk_begin;
  const TcChunk* const ch = chunks + tile.chunk_begin;

  if (warp < TC_GATHER_WARPS) {
    // gather warps: lanes l and l + 16 hold the map entry of row l of 16
    const int at = tile.row0 + warp * TC_WARP_ROWS + (lane & 15);
    const int row = at < out.rows ? __ldg(out.order + at) : -1;
    auto map_entry = [&](const TcChunk& c) { return row >= 0 ? (c.map ? __ldg(c.map + row) : (row << 1)) : -1; };
    uint4 pre[PARTS * MAXKQ / 2];
    auto load = [&](const TcChunk& c, int mp) {
      const int rb = c.xstride * ELEM;
      by_width<STEP, STEP, MAXKQ>(c.kpad * ELEM / 16, [&](auto kq) {
        Gather<decltype(kq)::value, SPLIT>::template load<ELEM>(pre, c.X, rb, mp, lane);
      });
    };
    TcChunk c, cn, cnn;
    int mp = -1, mp_next = -1;
    if (nchunks > 0) { c = ch[0]; mp = map_entry(c); }
    if (nchunks > 1) { cn = ch[1]; mp_next = map_entry(cn); }
    if (nchunks > 2) cnn = ch[2];
    if (nchunks > 0) load(c, mp);
    for (int j = 0; j < nchunks; ++j) {
      const int b = j & 1;
      uint8_t* const A = smem + b * a_bytes;
      // the MMAs that read this A stage (chunk j - 2) are done
      const bool free = j < 2 || mbar_wait(smem_u32(&mbar[b]), (uint32_t)((j >> 1) - 1) & 1u, polls);
      if (!__all_sync(0xffffffffu, free)) {
        s_fail = 1;
        break;
      }
      by_width<STEP, STEP, MAXKQ>(c.kpad * ELEM / 16,
                                  [&](auto kq) { Gather<decltype(kq)::value, SPLIT>::store(A, pre, warp, lane); });
      asm volatile("fence.proxy.async.shared::cta;");
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&mbar[3 + b])) : "memory");
      // rows of the next chunk, map of the one after, description of the third
      c = cn;
      mp = mp_next;
      if (j + 1 < nchunks) load(c, mp);
      cn = cnn;
      if (j + 2 < nchunks) mp_next = map_entry(cn);
      if (j + 3 < nchunks) cnn = ch[j + 3];
    }
  } else if (lane == 0) {
    // the issuing thread: B copies, MMAs, commits
    // idesc: D = F32, A/B = BF16 (kind::f16) or TF32 (kind::tf32), both K-major, M = 128
    uint32_t idesc = (1u << 4) | ((uint32_t)(out.npad >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    idesc |= ELEM == 4 ? ((2u << 7) | (2u << 10)) : ((1u << 7) | (1u << 10));
    auto copy_b = [&](int j) {
      const int st = j % b_stages;
      const uint32_t bar = smem_u32(&mbar[5 + st]);
      const uint32_t bytes = (uint32_t)(out.npad * ch[j].kpad * ELEM * PARTS);
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                       smem_u32(B0 + st * b_bytes)),
                   "l"(ch[j].W), "r"(bytes), "r"(bar)
                   : "memory");
    };
    const int ahead = b_stages - 2;   // B copies run this many chunks ahead
    int copies = 0;
    bool fail = false;
    for (; copies < ahead && copies < nchunks; ++copies) copy_b(copies);
    for (int j = 0; j < nchunks; ++j) {
      const int b = j & 1, st = j % b_stages;
      // chunk j - 2 read the stage that the next copy takes
      if (j >= 2 && !mbar_wait(smem_u32(&mbar[b]), (uint32_t)((j >> 1) - 1) & 1u, polls)) { fail = true; break; }
      if (copies < nchunks) copy_b(copies++);
      if (!mbar_wait(smem_u32(&mbar[3 + b]), (uint32_t)(j >> 1) & 1u, polls) ||
          !mbar_wait(smem_u32(&mbar[5 + st]), (uint32_t)(j / b_stages) & 1u, polls)) {
        fail = true;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;");
      const int kq = ch[j].kpad * ELEM / 16;
      const uint32_t sbo = (uint32_t)(kq * PARTS) * 128u;
      const uint64_t ad = smem_desc(smem_u32(smem + b * a_bytes), 128, sbo);
      const uint64_t bd = smem_desc(smem_u32(B0 + st * b_bytes), 128, sbo);
      // a K step is two core matrices: 256 bytes, 16 in the descriptor
      if (!SPLIT) {
        for (int ks = 0; ks < kq / 2; ++ks)
          mma<ELEM>(tmem, ad + ks * 16, bd + ks * 16, idesc, (j > 0 || ks > 0) ? 1u : 0u);
      } else {
        // x_hi W_hi + x_hi W_lo + x_lo W_hi; A and B tiles hold [hi | lo]
        for (int g = 0; g < 3; ++g) {
          const int pa = g == 2 ? kq * 8 : 0, pb = g == 1 ? kq * 8 : 0;
          for (int ks = 0; ks < kq / 2; ++ks)
            mma<ELEM>(tmem, ad + pa + ks * 16, bd + pb + ks * 16, idesc, (j > 0 || g > 0 || ks > 0) ? 1u : 0u);
        }
      }
      tc_commit(smem_u32(&mbar[b]));
    }
    // drain: one more commit arrives on mbar[2] once every MMA issued has
    // completed; after a timeout the default bound, here and for the copies
    // whose wait was given up, so that TMEM and shared memory are read and
    // freed only when nothing is in flight
    tc_commit(smem_u32(&mbar[2]));
    if (!mbar_wait(smem_u32(&mbar[2]), 0, polls)) {
      fail = true;
      mbar_wait(smem_u32(&mbar[2]), 0);
    }
    if (fail) {
      s_fail = 1;
      for (int j = max(0, copies - b_stages); j < copies; ++j)
        mbar_wait(smem_u32(&mbar[5 + j % b_stages]), (uint32_t)(j / b_stages) & 1u);
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const bool ok = s_fail == 0;
  if (!ok && tid == 0) atomicExch(err, 1);
  // accumulator to shared memory (the A stages are free): warps w and w + 4
  // read TMEM lanes 32 (w % 4) .. + 31, alternate groups of 16 columns
  const int ld = out.npad + 1;
  float* const D = (float*)smem;
  for (int c0 = 16 * (warp >> 2); warp < TC_GATHER_WARPS && c0 < out.npad; c0 += 32) {
    uint32_t v[16];
    if (nchunks > 0) {
      const uint32_t taddr = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0;
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
          : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
            "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
          : "r"(taddr));
      asm volatile("tcgen05.wait::ld.sync.aligned;");
    }
    float* d = D + (32 * (warp & 3) + lane) * ld + c0;
#pragma unroll
    for (int j = 0; j < 16; ++j) d[j] = nchunks > 0 && ok ? __uint_as_float(v[j]) : 0.f;
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
  // lanes along the rows of y; the terms without environment factor are added
  // in FP64 and in their order.  Each row lists those of the first TC_ADDS that
  // reach it (factor, source row): most of its projectors do not.
  const int rows = min(128, out.rows - tile.row0), total = rows * out.n;
  const int n_add = out.add_end - out.add_begin, held = min(n_add, TC_ADDS);
  double* const F = (double*)(smem + ((size_t)128 * ld * 4 + 15) / 16 * 16);
  int* const S = (int*)(F + TC_ADDS * 128);
  int* const R = S + TC_ADDS * 128;
  int* const C = R + 128;
  auto source = [&](const TcAdd& a, int g) { return a.map ? __ldg(a.map + g) : (g << 1); };
  auto factor = [&](const TcAdd& a, int g, int src) {
    const double f = (src & 1) ? -a.alpha : a.alpha;
    return a.val ? f * __ldg(a.val + g) : f;
  };
  if (tid < rows) {
    const int g = __ldg(out.order + tile.row0 + tid);
    int src[TC_ADDS], c = 0;
#pragma unroll
    for (int i = 0; i < TC_ADDS; ++i) src[i] = i < held ? source(adds[out.add_begin + i], g) : -1;
#pragma unroll
    for (int i = 0; i < TC_ADDS; ++i)
      if (src[i] >= 0) {
        F[c * 128 + tid] = factor(adds[out.add_begin + i], g, src[i]);
        S[c * 128 + tid] = src[i] >> 1;
        ++c;
      }
    R[tid] = g;
    C[tid] = c;
  }
  __syncthreads();
  // such a term keeps the parent charge: all of them read the output's own sector
  const float* const X = n_add > 0 ? adds[out.add_begin].X32 : nullptr;
  const int ldx = n_add > 0 ? adds[out.add_begin].ld : 0;
  double* const y = out.y + y_shift;
  for (int e0 = tid; e0 < total; e0 += TC_UNROLL * TC_THREADS) {
    double acc[TC_UNROLL];
    int r[TC_UNROLL], n[TC_UNROLL], most = 0;
#pragma unroll
    for (int u = 0; u < TC_UNROLL; ++u) {
      const int e = min(e0 + u * TC_THREADS, total - 1);
      r[u] = out.n == 1 ? e : (int)__umulhi((unsigned)e, out.div);
      n[u] = e - r[u] * out.n;
      acc[u] = f2d_exact(D[r[u] * ld + n[u]]);
      most = max(most, C[r[u]]);
    }
    for (int i = 0; i < most; ++i) {
      float x[TC_UNROLL];
#pragma unroll
      for (int u = 0; u < TC_UNROLL; ++u)
        x[u] = i < C[r[u]] ? __ldg(X + (long long)S[i * 128 + r[u]] * ldx + n[u]) : 0.f;
#pragma unroll
      for (int u = 0; u < TC_UNROLL; ++u)
        if (i < C[r[u]]) acc[u] = fma(F[i * 128 + r[u]], f2d_exact(x[u]), acc[u]);
    }
    for (int i = held; i < n_add; ++i) {
      const TcAdd a = adds[out.add_begin + i];
#pragma unroll
      for (int u = 0; u < TC_UNROLL; ++u) {
        const int src = source(a, R[r[u]]);
        if (src >= 0)
          acc[u] = fma(factor(a, R[r[u]], src), f2d_exact(__ldg(X + (long long)(src >> 1) * ldx + n[u])), acc[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < TC_UNROLL; ++u)
      if (e0 + u * TC_THREADS < total) y[(long long)R[r[u]] * out.n + n[u]] = acc[u];
  }
}

// FP64 -> BF16, rounded once: the FP32 value rounded to odd (the last bit set
// when something was cut off) rounds to the same BF16 as the FP64 one.
static __device__ __noinline__ __nv_bfloat16 d2bf_cast(double d) { return __double2bfloat16(d); }
__device__ __forceinline__ __nv_bfloat16 d2bf(double d) {
  const unsigned top = (unsigned)__double2hiint(d) & 0x7fffffffu;
  if (top - (920u << 20) >= (230u << 20)) return d2bf_cast(d);   // the range of d2ff's short form
  const ff t = d2ff(d);   // hi cut at 24 bits, lo the rest
  return __float2bfloat16_rn(__uint_as_float(__float_as_uint(t.hi) | (t.lo != 0.f ? 1u : 0u)));
}

// Split operand: x = d in FP32, hi = x cut to the 11 bits that the TF32 units
// read, lo = d - hi rounded to FP32.  d - hi is formed as an integer in units of
// d's last place.
static __device__ __noinline__ void split_cast(double d, float& x, float& hi, float& lo) {
  x = (float)d;
  hi = tf32_hi(x);
  lo = (float)(d - (double)hi);
}
__device__ __forceinline__ void split_tf32(double d, float& x, float& hi, float& lo) {
  const unsigned h = (unsigned)__double2hiint(d), l = (unsigned)__double2loint(d);
  const unsigned top = h & 0x7fffffffu;
  if (top - (949u << 20) >= (201u << 20)) {   // outside 2^-74 .. 2^127
    if ((top | l) == 0u) {
      x = hi = lo = 0.f;
      return;
    }
    split_cast(d, x, hi, lo);
    return;
  }
  x = d2f_rn(d);
  hi = tf32_hi(x);
  const unsigned hb = __float_as_uint(hi) & 0x7fffffffu, e = top >> 20;   // hi's exponent is d's or one more
  const long long m = ((long long)((top & 0xfffffu) | 0x100000u) << 32) | l;
  const long long hm = (long long)((hb & 0x7fffffu) | 0x800000u) << (29 + (hb >> 23) - (e - 896u));
  const float r = __ll2float_rn(m - hm) * __uint_as_float((e - 948u) << 23);
  lo = (h >> 31) ? -r : r;
}

// One warp per padded row, lanes along the row: coalesced reads of the FP64
// source and writes of the FP32 copy and, for BF16 and split operands, of the
// operand rows.  Converted on the integer pipes: FP64 conversions run at the
// FP64 rate.
enum { CONV_F32 = 0, CONV_BF16 = 1, CONV_SPLIT = 2 };
template <int MODE>
__global__ void __launch_bounds__(256) convert_kernel(const ConvJob* __restrict__ jobs, long long shift) {
  const ConvJob j = jobs[blockIdx.y];
  const int lane = threadIdx.x & 31;
  const int warps = (int)(gridDim.x * (blockDim.x >> 5));
  const double* src = j.src + shift;
  for (int r = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 4; r < j.rows; r += warps * 4) {
    for (int c = lane; c < j.kpad; c += 32) {
      double x[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        x[i] = c < j.cols && r + i < j.rows ? __ldg(src + (long long)(r + i) * j.ld_src + c) : 0.0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (r + i >= j.rows) break;
        const long long e = (long long)(r + i) * j.kpad + c;
        if (MODE == CONV_SPLIT) {
          float* d = (float*)j.dst + (long long)(r + i) * 2 * j.kpad + c;
          split_tf32(x[i], j.dst32[e], d[0], d[j.kpad]);
        } else {
          j.dst32[e] = d2f_rn(x[i]);
          if (MODE == CONV_BF16) ((__nv_bfloat16*)j.dst)[e] = d2bf(x[i]);
        }
      }
    }
  }
}

// One environment block, scaled, as the B operand in core-matrix order (rows
// padded with zeros to npad, columns to kpad): BF16, TF32, or TF32 [hi | lo].
template <int ELEM, bool SPLIT>
__global__ void __launch_bounds__(256) stage_w_kernel(const WJob* __restrict__ jobs) {
  const WJob j = jobs[blockIdx.x];
  const int kq = j.kpad * ELEM / 16, kchunks = SPLIT ? 2 * kq : kq;
  uint8_t* dst = (uint8_t*)j.dst;
  for (int e = threadIdx.x; e < j.npad * j.kpad; e += blockDim.x) {
    const int n = e / j.kpad, k = e - n * j.kpad;
    const double v = n < j.rows && k < j.cols ? j.scale * j.src[(long long)n * j.ld_src + k] : 0.0;
    const int q = k * ELEM / 16, in = k * ELEM % 16;
    if (ELEM == 2) {
      *(__nv_bfloat16*)(dst + core_off(n, q, kchunks) + in) = __double2bfloat16(v);
    } else if (!SPLIT) {
      *(float*)(dst + core_off(n, q, kchunks) + in) = (float)v;
    } else {
      // hi = TF32-truncated, lo = FP32 residual
      const float hi = tf32_hi((float)v);
      *(float*)(dst + core_off(n, q, kchunks) + in) = hi;
      *(float*)(dst + core_off(n, kq + q, kchunks) + in) = (float)(v - (double)hi);
    }
  }
}

}  // namespace

int launch_tc_heff(int elem, int split, const TcTile* tiles, int n_tiles, const TcOutput* outs,
                   const TcChunk* chunks, const TcAdd* adds, int max_kpad, int max_npad, long long y_shift, int* err,
                   cudaStream_t s, long long polls) {
  if (n_tiles <= 0) return 0;
  if (polls < 0) polls = kWaitPolls;
  const int parts = split ? 2 : 1;
  const int a_bytes = 128 * max_kpad * parts * elem;
  const int b_bytes = max_npad * max_kpad * parts * elem;
  if (2 * (a_bytes + b_bytes) > 200 * 1024 || max_npad > 256 || max_npad % 16 || max_kpad % 16) return -7;
  if (split && elem != 4) return -7;
  // three or four B stages where that costs no CTA of the SM
  const int sm = 226 * 1024, fit = std::max(1, sm / (2 * (a_bytes + b_bytes) + 1024));
  int b_stages = 2;
  while (b_stages < 4 && sm / (2 * a_bytes + (b_stages + 1) * b_bytes + 1024) >= std::min(fit, 2)) ++b_stages;
  const int smem = std::max(2 * a_bytes + b_stages * b_bytes, 128 * (max_npad + 1) * 4 + 16 + TC_ADDS * 128 * 12 + 2 * 128 * 4);
  auto pick = [&](auto type, auto is_split) {
    constexpr int E = decltype(type)::value;
    constexpr bool S = decltype(is_split)::value;
    using W = Width<E, S>;
    return max_kpad * E / 16 <= W::NARROW ? tc_heff_kernel<E, S, W::NARROW> : tc_heff_kernel<E, S, W::WIDE>;
  };
  using Two = std::integral_constant<int, 2>;
  using Four = std::integral_constant<int, 4>;
  auto kern = elem == 2 ? pick(Two(), std::false_type()) : (split ? pick(Four(), std::true_type()) : pick(Four(), std::false_type()));
  if (max_kpad * elem / 16 > (elem == 2 ? Width<2, false>::WIDE : (split ? Width<4, true>::WIDE : Width<4, false>::WIDE))) return -7;
  allow_smem((const void*)kern, 226 * 1024);
  kern<<<n_tiles, TC_THREADS, smem, s>>>(tiles, outs, chunks, adds, a_bytes, b_bytes, b_stages, y_shift, err, polls);
  count_launches(1);
  return 0;
}

void launch_convert(int elem, int split, const ConvJob* jobs, int n_jobs, long long max_elems, long long shift,
                    cudaStream_t s) {
  if (n_jobs <= 0) return;
  // rows <= max_elems / 16 (kpad >= 16); 32 rows per block, about 8 blocks per SM in total
  long long gx = (max_elems / 16 + 31) / 32;
  const long long cap = std::max(1LL, 1216LL / n_jobs);
  if (gx > cap) gx = cap;
  if (gx < 1) gx = 1;
  dim3 grid((unsigned)gx, (unsigned)n_jobs);
  if (elem == 2)
    convert_kernel<CONV_BF16><<<grid, 256, 0, s>>>(jobs, shift);
  else if (split)
    convert_kernel<CONV_SPLIT><<<grid, 256, 0, s>>>(jobs, shift);
  else
    convert_kernel<CONV_F32><<<grid, 256, 0, s>>>(jobs, shift);
  count_launches(1);
}

void launch_stage_w(int elem, int split, const WJob* jobs, int n_jobs, cudaStream_t s) {
  if (n_jobs <= 0) return;
  if (elem == 2)
    stage_w_kernel<2, false><<<n_jobs, 256, 0, s>>>(jobs);
  else if (split)
    stage_w_kernel<4, true><<<n_jobs, 256, 0, s>>>(jobs);
  else
    stage_w_kernel<4, false><<<n_jobs, 256, 0, s>>>(jobs);
  count_launches(1);
}

}  // namespace qed
