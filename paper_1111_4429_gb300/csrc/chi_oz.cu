// Plain-precision (FP64) polarizability on the 5th-generation tensor cores
// (paper, Eq. eqn_static_xi as the matrix product of Eq.
// eqn_static_xi_compact), by an error-free splitting of the operands (the
// Ozaki scheme):
//
//   X[p][G] = M[p][G] sqrt|w_p|  (w_p < 0 always: the sign is pulled out)
//   chi[G][G'] (+)= -(4/Omega) sum_p conj(X[p][G]) X[p][G']
//
// Every column G is scaled by the power of two 2^e_G above its largest entry
// over all pairs and cut into S = 8 digits of 7 bits,
//   X = 2^e sum_a 2^{-7(a+1)} h_a,  |h_0| <= 128, |h_a| <= 64,
// integers that FP16 holds exactly.  The products of digits a and b belong to
// level L = a + b; the tensor cores' FP32 sums of one level over a segment of
// kSegStages stages (384 real products per digit pair) stay below 2^24
// (2^14 + 6 2^12 times 384 at the deepest level), so they are exact.  Levels
// 0 .. 7 are kept (36 digit products); a segment's eight sums are joined in
// integers and added to two 64-bit integers per value, without rounding, and
// converted to FP64 once per CTA.  What is lost are the bits of X below
// 2^(e - 56) and the levels past 7: an error near 2^-58 sqrt(6 K) 2^(e_G + e_G'),
// against 2^-53 0.3 sqrt(K) |chi| of a running FP64 sum (chi_f64_kernel); the
// running sum's error grows with K, this one's relative size does not.  The
// bound is relative to (chi_GG chi_G'G')^1/2; for it to hold for every block of
// chi as well, the pairs' sizes may not spread too far (kSpreadBits).
//
// Why: the SM's FP64 pipe (2 FMA per clock) bounds chi_f64_kernel at
// 1.12 TFLOP/s; 36 exact FP16 products per FP64 one on the tensor cores are
// far cheaper.  One CTA = one 128 x 32 tile and one group of segments: 16
// accumulators (8 levels, Re and Im) of 32 columns fill tensor memory.  The
// digits of the 32-column operand lie one after the other in shared memory,
// so digit a of the row operand takes one MMA of N = 32 (8 - a) columns.
// Shared memory: a three-deep ring of row-operand stages (64 KB: 8 digits x
// 128 rows x 16 pairs) and a two-deep one of column-operand stages (16 KB).
//
// Bound by the tensor pipe (62 % active at N_G 2120, K 6400, 3.29 ms): one set of
// level sums fills tensor memory, so between two segments it waits for them to be
// read and joined (issue slots 9 %, ALU 7 %, L2 hits 83 %).
//
// Measured (N_G 2120): K 25600 in 13.8 ms per call (412 ms by chi_f64_kernel),
// of it 12.7 ms here and 0.9 ms for the maximum and digit passes; K 2400 in
// 1.5 ms (38.6 ms).  Relative error against quad-precision sums, off-diagonal /
// diagonal: 6.6e-16 / 2.0e-16 at K 25600 (FMA kernel 4.1e-15 / 3.0e-15),
// 1.6e-16 / 1.0e-16 at K 2400 (7.7e-16 / 1.9e-15).
//
// A column with an infinity or NaN cannot be scaled, and pairs of very different
// sizes lose bits: the maximum pass then sets a device flag, the kernels here
// return and chi_f64_kernel, launched behind the same flag, does the call.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <vector>

#include "runtime.h"
#include "sweep_common.cuh"
#include "tc_common.cuh"

namespace bgw {

namespace oz64 {

using tc::BM;
constexpr int BN = 32;           // tile columns
constexpr int S = 8;             // digits per value
constexpr int BETA = 7;          // bits per digit
constexpr int SK = 32;           // real values per row and stage (16 complex pairs: 16 Re, 16 Im)
constexpr int kSegStages = 12;   // stages summed exactly in FP32
constexpr int kUPlane = BM * SK * 2;          // 8 KiB
constexpr int kVPlane = BN * SK * 2;          // 2 KiB
constexpr int kUStage = S * kUPlane, kVStage = S * kVPlane;
constexpr int kURing = 3, kVRing = 2;
constexpr int kEpiWarps = 8;
constexpr int kThreads = 32 * (kEpiWarps + 2);
constexpr size_t kSmem = (size_t)kURing * kUStage + (size_t)kVRing * kVStage + 1024 + 256;
static_assert(kSmem <= 227 * 1024, "shared memory of one CTA");
constexpr int kTileElems = BM * BN;

// Operand values of pair p and column g, as the maximum and digit passes read
// them.  kHerm: M sqrt|w| (complex), kReal: the same with real M, kWeighted:
// M w / sqrt|w| with complex w (against kHerm: a resonance's weight is shared
// by both operands, so that neither spreads over the pairs more than its root).
enum Operand { kHerm = 0, kReal = 1, kWeighted = 2 };

template <int OP>
__device__ __forceinline__ double2 operand(const void* __restrict__ M, const double* __restrict__ fac,
                                           const double2* __restrict__ wc, long long p, int g, int ng) {
  if constexpr (OP == kReal) {
    return make_double2(static_cast<const double*>(M)[p * ng + g] * fac[p], 0.0);
  } else {
    const double2 m = static_cast<const double2*>(M)[p * ng + g];
    if constexpr (OP == kHerm) {
      const double s = fac[p];
      return make_double2(m.x * s, m.y * s);
    } else {
      const double2 w = wc[p];
      return make_double2(fma(w.x, m.x, -w.y * m.y), fma(w.x, m.y, w.y * m.x));
    }
  }
}

// Size of a value as an integer that orders as its binary exponent: 0 for zero,
// 1 below the normal range, then the exponent field + 1; kNotFinite for an
// infinity or NaN.
constexpr int kNotFinite = 0x800;
__device__ __forceinline__ int size_of(double x) {
  const unsigned hi = (unsigned)__double2hiint(x) & 0x7FFFFFFFu;
  return (hi | (unsigned)__double2loint(x)) ? (int)(hi >> 20) + 1 : 0;
}
// Scale exponent of a column from its largest size: |x| 2^-e < 1.
__device__ __forceinline__ int scale_of(int size) { return size ? size - 1023 : 0; }

// A column's scale is set by its largest entry over all pairs, so a pair 2^s
// smaller than the largest one keeps s bits less of its operands.  Norm-wise
// nothing is lost, but blocks of chi that only the smaller pairs make are.
// Sizes of the pairs (their largest operand) further apart than 2^kSpreadBits
// leave the call to the FMA kernels.  Blocks made by pairs 2^s below the largest
// one, relative error here / in running sums: K 240, s 6 / 8 / 12 / 20: 4.9e-16,
// 1.7e-15, 2.8e-14, 6.6e-12 / 5.5e-16; K 2400: 5e-16, 1.6e-15, 2.1e-14, 7.5e-12 /
// 1.7e-15.  Pairs of one band structure lie within 2^7: sqrt|w| over gaps of 0.04
// to 2 Ha 2^2.8, on the real axis (broadening 0.02 and more) 2^5, elements 2^2.
constexpr int kSpreadBits = 8;

// sqrt|w|, and for complex weights w / sqrt|w|.
__global__ void sqrt_weights_kernel(const double* __restrict__ w, const double2* __restrict__ wc, long long K,
                                    double* __restrict__ out, double2* __restrict__ outc) {
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= K) return;
  if (!wc) {
    out[p] = sqrt(fabs(w[p]));
    return;
  }
  const double2 z = wc[p];
  const double s = sqrt(hypot(z.x, z.y));
  out[p] = s;
  outc[p] = s > 0.0 ? make_double2(z.x / s, z.y / s) : z;
}

// Sizes of one operand, zeroed before the pass that fills them: of each
// column, of each pair, and how many CTAs are done.
struct Sizes {
  int* col;
  int* pair;
  int* done;
};

// sz.col[g] = largest size over the pairs, sz.pair[p] = largest size over the
// columns; *flag = 1 where a value is not finite or, found by the last CTA, the
// pairs' sizes spread by more than kSpreadBits.  One pass over M.  grid
// (ceil(ng/64), strips of pairs), block 256 = 64 columns x 4 pairs.  N_G 2120, 6400
// pairs: 84 us, 2.6 TB/s, half the warps resident and the FP64 products 60 % of
// their pipe (the pairs' sizes add 9 us to a call of 2400 pairs, 1453 -> 1461 us).
template <int OP>
__global__ void __launch_bounds__(256) colmax_kernel(const void* __restrict__ M, const double* __restrict__ fac,
                                                     const double2* __restrict__ wc, long long K, int ng,
                                                     const Sizes sz, int* __restrict__ flag) {
  __shared__ int red[4][64];
  __shared__ int lohi[2], last;
  const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
  const int g = blockIdx.x * 64 + tx;
  int m = 0;
#pragma unroll 4
  for (long long p = (long long)blockIdx.y * 4 + ty; p < K; p += 4LL * gridDim.y) {   // a warp has one pair
    int k = 0;
    if (g < ng) {
      const double2 v = operand<OP>(M, fac, wc, p, g, ng);
      k = max(size_of(v.x), size_of(v.y));
    }
    m = max(m, k);
    const int row = __reduce_max_sync(0xffffffffu, k);
    if ((tx & 31) == 0 && row) atomicMax(sz.pair + p, row);
  }
  red[ty][tx] = m;
  __syncthreads();
  if (ty == 0 && g < ng) {
    m = max(max(red[0][tx], red[1][tx]), max(red[2][tx], red[3][tx]));
    if (m) atomicMax(sz.col + g, m);
    if (m == kNotFinite) atomicExch(flag, 1);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(sz.done, 1) == (int)(gridDim.x * gridDim.y) - 1;
    lohi[0] = kNotFinite;
    lohi[1] = 0;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  int lo = kNotFinite, hi = 0;   // over the pairs that are not zero
#pragma unroll 8
  for (long long p = threadIdx.x; p < K; p += 256) {
    const int k = __ldcg(sz.pair + p);
    if (k) lo = min(lo, k);
    hi = max(hi, k);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&lohi[0], lo);
    atomicMax(&lohi[1], hi);
  }
  __syncthreads();
  if (threadIdx.x == 0 && lohi[1] - lohi[0] > kSpreadBits) atomicExch(flag, 1);
}

// Digit a of two adjacent values (X0, X1: rint(x 2^(56 - e))) as a half2:
// balanced base-128 digits, integer arithmetic only.  0x6400 + d + 512 are
// the FP16 bits of 1536 + d exactly (unit spacing in [1024, 2048)).
__device__ __forceinline__ void store_digits(long long X0, long long X1, __half* out, size_t plane) {
  __half2 h[S];
#pragma unroll
  for (int a = S - 1; a >= 0; --a) {
    int d0, d1;
    if (a > 0) {
      d0 = (int)((X0 + 64) & 127) - 64;
      d1 = (int)((X1 + 64) & 127) - 64;
      X0 = (X0 - d0) >> BETA;
      X1 = (X1 - d1) >> BETA;
    } else {
      d0 = (int)X0;
      d1 = (int)X1;
    }
    const unsigned u = ((unsigned)(0x6600 + d0) & 0xFFFFu) | ((unsigned)(0x6600 + d1) << 16);
    h[a] = __hsub2(*reinterpret_cast<const __half2*>(&u), __half2half2(__ushort_as_half(0x6600)));
  }
#pragma unroll
  for (int a = 0; a < S; ++a) *reinterpret_cast<__half2*>(out + a * plane) = h[a];
}

// Digits of the pairs p0 .. p0 + K - 1 (padded with zeros to whole stages) of
// every column, K-major: planes[a][g][...], a stage's 32 values being 16 real
// and 16 imaginary parts of 16 pairs (kReal: 32 pairs).  32 x 32 tiles
// transposed in shared memory; 16 bytes read and 32 written per value.  N_G 2120,
// 6400 pairs: 151 us, 4.0 TB/s, bound by the integer pipe (80 %).  grid
// (ceil(kpad/32), rows/32), block 256.
template <int OP>
__global__ void __launch_bounds__(256) digits_kernel(const void* __restrict__ M, const double* __restrict__ fac,
                                                     const double2* __restrict__ wc, long long p0, long long K,
                                                     int ng, int rows, size_t rowlen, const int* __restrict__ field,
                                                     const int* __restrict__ flag, __half* __restrict__ planes) {
  constexpr bool real = OP == kReal;
  __shared__ long long xr[32][33];
  __shared__ long long xi[real ? 1 : 32][33];
  if (*flag) return;
  const long long pc0 = (long long)blockIdx.x * 32;
  const int g0 = blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int e = g0 + tx < ng ? scale_of(field[g0 + tx]) : 0;
#pragma unroll
  for (int r = ty; r < 32; r += 8) {
    double2 v = make_double2(0.0, 0.0);
    if (pc0 + r < K && g0 + tx < ng) v = operand<OP>(M, fac, wc, p0 + pc0 + r, g0 + tx, ng);
    xr[r][tx] = fixed56(v.x, e);
    if constexpr (!real) xi[r][tx] = fixed56(v.y, e);
  }
  __syncthreads();
  const size_t plane = (size_t)rows * rowlen;
  if constexpr (real) {
    const int half = tx >> 4, pp = 2 * (tx & 15);
    for (int gr = 2 * ty + half; gr < 32; gr += 16)
      store_digits(xr[pp][gr], xr[pp + 1][gr], planes + (size_t)(g0 + gr) * rowlen + pc0 + pp, plane);
  } else {
    // lane: values 2 lane, 2 lane + 1 of the row's 64: pair 16 (lane / 16) + 2 (lane % 8), Re or Im by bit 3
    const int pp = (tx >> 4) * 16 + 2 * (tx & 7);
    if (2 * pc0 + 2 * tx >= (long long)rowlen) return;   // odd number of stages: the last tile is half a tile
    for (int gr = ty; gr < 32; gr += 8) {
      const bool im = (tx & 8) != 0;
      const long long a = im ? xi[pp][gr] : xr[pp][gr], b = im ? xi[pp + 1][gr] : xr[pp + 1][gr];
      store_digits(a, b, planes + (size_t)(g0 + gr) * rowlen + 2 * pc0 + 2 * tx, plane);
    }
  }
}

// Digits of row-major operands (the Sigma forms): src[r][k] complex, rows
// r < R, the K inner values of a row in stages as above; conj negates the
// imaginary parts.  One warp per row: its largest exponent, then its digits.
__global__ void __launch_bounds__(256) row_digits_kernel(const double2* __restrict__ src, int R, int K, int rows,
                                                         size_t rowlen, int conj, int* __restrict__ field,
                                                         int* __restrict__ flag, __half* __restrict__ planes) {
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= rows) return;
  int m = 0;
  if (r < R)
    for (int k = lane; k < K; k += 32) {
      const double2 v = src[(size_t)r * K + k];
      m = max(m, max(size_of(v.x), size_of(v.y)));
    }
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) {
    field[r] = m;
    if (m == kNotFinite) atomicExch(flag, 1);
  }
  if (m == kNotFinite) m = 0;   // the product is not used
  const int e = scale_of(m);
  const size_t plane = (size_t)rows * rowlen;
  for (size_t x = 0; x < rowlen; x += 64) {
    // values 2 lane, 2 lane + 1 of this 64: inner index, Re or Im by bit 3 of the lane
    const int k = (int)(x / 2) + (lane >> 4) * 16 + 2 * (lane & 7);
    if (x + 2 * lane >= rowlen) break;
    double v[2] = {0.0, 0.0};
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (r < R && k + q < K) {
        const double2 z = src[(size_t)r * K + k + q];
        v[q] = (lane & 8) ? (conj ? -z.y : z.y) : z.x;
      }
    store_digits(fixed56(v[0], e), fixed56(v[1], e), planes + (size_t)r * rowlen + x + 2 * lane, plane);
  }
}

// Packed joint value of a segment's level pair: s0 2^7 + s1 (|.| < 2^31).
__device__ __forceinline__ int join(uint32_t s0, uint32_t s1) {
  return __float2int_rn(__uint_as_float(s0)) * (1 << BETA) + __float2int_rn(__uint_as_float(s1));
}

// One CTA: tile (tiles[t]) x group of stages [grp segs seg_stages, ...) of
//   C[i][j] = sum_p conj(U[p][i]) V[p][j]
// as a double2 partial work[grp][t][128][32] (REALV: imaginary parts zero).
// The pipeline, its bounded waits and the give-up path are those of
// chi_tc_kernel.
template <bool REALV>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_kernel(const __grid_constant__ CUtensorMap umap, const __grid_constant__ CUtensorMap vmap, int urows,
                int vrows, int nstages, int seg_stages, int segs, int ntiles, const int2* __restrict__ tiles,
                const int* __restrict__ ufield, const int* __restrict__ vfield, const int* __restrict__ flag,
                unsigned long long wait_ns, double2* __restrict__ work, int* __restrict__ status) {
  using namespace tc;
  using oz64::kThreads;
  if (*flag) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* us = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* vs = us + kURing * kUStage;
  uint64_t* ufull = reinterpret_cast<uint64_t*>(vs + kVRing * kVStage);
  uint64_t* uempty = ufull + kURing;
  uint64_t* vfull = uempty + kURing;
  uint64_t* vempty = vfull + kVRing;
  uint64_t* done = vempty + kVRing;
  uint64_t* tfree = done + 1;
  uint64_t* mflush = tfree + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mflush + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = blockIdx.x / ntiles, tix = blockIdx.x - grp * ntiles;
  const int2 tile = tiles[tix];
  const int row0 = tile.x * BM, col0 = tile.y * BN;
  const int s0 = grp * segs * seg_stages;
  const int nk = max(0, min(nstages, s0 + segs * seg_stages) - s0);
  const int nseg = (nk + seg_stages - 1) / seg_stages;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kURing; ++s) {
      mbar_init(&ufull[s], 1);
      mbar_init(&uempty[s], 1);
    }
    for (int s = 0; s < kVRing; ++s) {
      mbar_init(&vfull[s], 1);
      mbar_init(&vempty[s], 1);
    }
    mbar_init(done, 1);
    mbar_init(tfree, kEpiWarps);
    mbar_init(mflush, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kEpiWarps) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;   // Re of level L in columns 32 L, Im in 256 + 32 L

  if (warp == kEpiWarps) {
    if (lane == 0) {
      // ---------------- TMA producer
      int issued = 0;
      for (int i = 0; i < nk; ++i) {
        const int su = i % kURing, sv = i % kVRing;
        if ((i >= kURing && !mbar_wait(&uempty[su], (i / kURing - 1) & 1, abort_flag, wait_ns)) ||
            (i >= kVRing && !mbar_wait(&vempty[sv], (i / kVRing - 1) & 1, abort_flag, wait_ns))) {
          if (!*abort_flag) atomicExch(status, (int)kDevTimeout);
          *abort_flag = 1;
          break;
        }
        const int x = (s0 + i) * SK;
        mbar_expect_tx(&vfull[sv], kVStage);
        for (int a = 0; a < S; ++a)
          tma_load_2d(vs + sv * kVStage + a * kVPlane, &vmap, &vfull[sv], x, a * vrows + col0);
        mbar_expect_tx(&ufull[su], kUStage);
        for (int a = 0; a < S; ++a)
          tma_load_2d(us + su * kUStage + a * kUPlane, &umap, &ufull[su], x, a * urows + row0);
        issued = i + 1;
      }
      // no copies in flight at exit (bounded)
      for (int i = max(0, issued - kURing); i < issued; ++i) {
        const uint64_t t0 = globaltimer();
        while (!mbar_try_wait(&ufull[i % kURing], (i / kURing) & 1) && globaltimer() - t0 < kWaitNs) {
        }
      }
      for (int i = max(0, issued - kVRing); i < issued; ++i) {
        const uint64_t t0 = globaltimer();
        while (!mbar_try_wait(&vfull[i % kVRing], (i / kVRing) & 1) && globaltimer() - t0 < kWaitNs) {
        }
      }
    }
  } else if (warp == kEpiWarps + 1) {
    if (lane == 0) {
      // ---------------- MMA issuer
      bool ok = true;
      for (int i = 0; i < nk && ok; ++i) {
        const int su = i % kURing, sv = i % kVRing, kin = i % seg_stages;
        if (kin == 0 && i > 0) {
          // the previous segment's sums must have left tensor memory
          if (!mbar_wait(tfree, (i / seg_stages - 1) & 1, abort_flag, wait_ns)) {
            ok = false;
            break;
          }
          fence_after();
        }
        if (!mbar_wait(&vfull[sv], (i / kVRing) & 1, abort_flag, wait_ns) ||
            !mbar_wait(&ufull[su], (i / kURing) & 1, abort_flag, wait_ns)) {
          ok = false;
          break;
        }
        fence_after();
        const uint64_t du = sdesc(smem_u32(us + su * kUStage)), dv = sdesc(smem_u32(vs + sv * kVStage));
        // Re, Im: the row's 16 real parts, then its 16 imaginary parts 32 bytes on (+2 in the descriptor)
#pragma unroll
        for (int a = 0; a < S; ++a) {
          const uint32_t dre = tmem + BN * a, dim = tmem + BN * (S + a);
          const uint64_t ua = du + (uint64_t)((a * kUPlane) >> 4);
          const uint32_t id = idesc(BN * (S - a), false, false), idn = idesc(BN * (S - a), false, true);
          // level L is first written by digit a = 0
          const uint32_t acc0 = (a > 0 || kin > 0) ? 1u : 0u;
          mma(dre, ua, dv, id, acc0);              // Re = ur vr + ui vi
          mma(dre, ua + 2, dv + 2, id, 1u);
          if constexpr (!REALV) {
            mma(dim, ua, dv + 2, id, acc0);        // Im = ur vi - ui vr
            mma(dim, ua + 2, dv, idn, 1u);
          }
        }
        mma_commit(&uempty[su]);
        mma_commit(&vempty[sv]);
        if (kin == seg_stages - 1 || i == nk - 1) mma_commit(done);
      }
      if (!ok) {
        // let the issued MMAs finish, then wake the epilogue (it sees the abort flag)
        mma_commit(mflush);
        const uint64_t t0 = globaltimer();
        while (!mbar_try_wait(mflush, 0) && globaltimer() - t0 < kWaitNs) {
        }
        if (!*abort_flag) atomicExch(status, (int)kDevTimeout);
        *abort_flag = 1;
        mma_commit(done);
      }
    }
  } else {
    // ---------------- epilogue: row 32 (warp % 4) + lane, 16 columns from 16 (warp / 4)
    constexpr int HC = BN / 2, NPART = REALV ? 1 : 2;
    const int q = warp & 3, h = warp >> 2;
    const uint32_t lane_off = ((uint32_t)(q * 32) << 16) + (uint32_t)(h * HC);
    // level sums joined as hi (levels 0..3, unit 2^-35) and lo (levels 4..7, unit 2^-63)
    long long hi[NPART][HC], lo[NPART][HC];
#pragma unroll
    for (int k = 0; k < NPART; ++k)
#pragma unroll
      for (int j = 0; j < HC; ++j) hi[k][j] = lo[k][j] = 0;
    bool have = true;
    for (int sg = 0; sg < nseg; ++sg) {
      bool got = mbar_wait(done, sg & 1, abort_flag, kWaitNs, false);
      got = __all_sync(0xffffffffu, got) != 0;
      if (!got) {
        if (lane == 0 && !*abort_flag) atomicExch(status, (int)kDevTimeout);
        *abort_flag = 1;
      }
      if (!got || __any_sync(0xffffffffu, *abort_flag != 0)) {
        have = false;
        break;
      }
      fence_after();
#pragma unroll
      for (int k = 0; k < NPART; ++k)
#pragma unroll
        for (int c0 = 0; c0 < HC; c0 += 4) {
          uint32_t x[S][4];
#pragma unroll
          for (int L = 0; L < S; ++L) tmem_ld4(tmem + lane_off + BN * (k * S + L) + c0, x[L]);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            hi[k][c0 + j] += (long long)join(x[0][j], x[1][j]) * (1LL << (2 * BETA)) + join(x[2][j], x[3][j]);
            lo[k][c0 + j] += (long long)join(x[4][j], x[5][j]) * (1LL << (2 * BETA)) + join(x[6][j], x[7][j]);
          }
        }
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tfree);
    }
    if (have) {
      const int row = q * 32 + lane;
      const int eu = scale_of(ufield[row0 + row]);
      double2* w = work + ((size_t)grp * ntiles + tix) * kTileElems + (size_t)row * BN + h * HC;
#pragma unroll
      for (int j = 0; j < HC; ++j) {
        const int ex = eu + scale_of(vfield[col0 + h * HC + j]);
        double v[2] = {0.0, 0.0};
#pragma unroll
        for (int k = 0; k < NPART; ++k)
          v[k] = ldexp(fma((double)lo[k][j], 0x1p-28, (double)hi[k][j]), ex - 5 * BETA);
        w[j] = make_double2(v[0], v[1]);
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == kEpiWarps) {
    __syncwarp();
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

// chi[g][g'] (+)= factor sum_groups work.  HERM: lower triangle, mirrored
// (conjugated) into the upper one; REALV: the same with real chi; else every
// element.  One thread per tile element.
template <bool HERM, bool REALV>
__global__ void reduce_kernel(const double2* __restrict__ work, int ngroups, int ntiles,
                              const int2* __restrict__ tiles, int ng, double factor, int accumulate,
                              const int* __restrict__ flag, void* __restrict__ chi) {
  if (*flag) return;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)ntiles * kTileElems) return;
  const int tix = (int)(e / kTileElems), k = (int)(e % kTileElems);
  const int2 tl = tiles[tix];
  const int g = tl.x * BM + k / BN, gp = tl.y * BN + k % BN;
  if (g >= ng || gp >= ng || (HERM && gp > g)) return;
  double2 s = work[e];
  for (int q = 1; q < ngroups; ++q) {
    const double2 t = work[(size_t)q * ntiles * kTileElems + e];
    s.x += t.x;
    s.y += t.y;
  }
  const size_t lo = (size_t)g * ng + gp, up = (size_t)gp * ng + g;
  if constexpr (REALV) {
    double* c = static_cast<double*>(chi);
    double v = s.x * factor;
    if (accumulate) v += c[lo];
    c[lo] = v;
    if (g != gp) c[up] = v;
  } else {
    double2* c = static_cast<double2*>(chi);
    double2 v = make_double2(s.x * factor, s.y * factor);
    if (accumulate) {
      const double2 o = c[lo];
      v.x += o.x;
      v.y += o.y;
    }
    if (HERM && g == gp) v.y = 0.0;
    c[lo] = v;
    if (HERM && g != gp) c[up] = make_double2(v.x, -v.y);
  }
}

// The Sigma forms of pair p = p0 + i, one warp per pair: C = W m from the
// product's partial tiles, qW = Re sum_G conj(m_p(G)) C(G), qV = sum_G |m_p(G)|^2 v_G.
__global__ void __launch_bounds__(256) sigma_forms_kernel(const double2* __restrict__ M, long long p0, int R, int ng,
                                                          const double* __restrict__ sv,
                                                          const double2* __restrict__ work, int ngroups, int ntiles,
                                                          const int* __restrict__ flag, double* __restrict__ qW,
                                                          double* __restrict__ qV) {
  if (*flag) return;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= R) return;
  const int nJ = (ng + BN - 1) / BN;
  const double2* m = M + (p0 + i) * ng;
  double w = 0.0, s = 0.0;
  for (int J = 0; J < nJ; ++J) {
    const int g = J * BN + lane;
    if (g >= ng) break;
    const double2* t = work + ((size_t)(i / BM) * nJ + J) * kTileElems + (size_t)(i % BM) * BN + lane;
    double2 c = *t;
    for (int q = 1; q < ngroups; ++q) {
      const double2 x = t[(size_t)q * ntiles * kTileElems];
      c.x += x.x;
      c.y += x.y;
    }
    const double2 v = m[g];
    w = fma(v.x, c.x, fma(v.y, c.y, w));
    s = fma(fma(v.x, v.x, v.y * v.y), sv[g] * sv[g], s);
  }
  for (int o = 16; o > 0; o >>= 1) {
    w += __shfl_xor_sync(0xffffffffu, w, o);
    s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  if (lane == 0) {
    qW[p0 + i] = w;
    qV[p0 + i] = s;
  }
}

}  // namespace oz64

namespace {
// Operand digits of one chunk of pairs: 32 bytes per complex value and
// operand.  Longer calls go chunk by chunk, each chunk's FP64 sum added into
// chi.  Where the pool cannot give the whole size (a small budget) the chunk
// is halved, down to kMinChunk pairs; below that the caller's FP64 FMA kernel
// takes the call.
constexpr size_t kOzChunkBytes = size_t(1) << 30;
constexpr long long kMinChunk = 512;

template <int OP>
void launch_colmax(Ctx* c, const void* M, const double* fac, const double2* wc, long long K, int ng,
                   const oz64::Sizes& sz, int* flag, cudaStream_t st) {
  const int gx = (ng + 63) / 64;
  const int gy = (int)std::min<long long>((K + 3) / 4, std::max(1, sm_count(c) * 8 / gx));
  oz64::colmax_kernel<OP><<<dim3(gx, gy), 256, 0, st>>>(M, fac, wc, K, ng, sz, flag);
}
}  // namespace

// Digit planes, exponents and partial sums of one product.
struct OzGemm {
  int urows = 0, vrows = 0;
  long long kpad = 0;        // inner values (pairs) the planes hold
  size_t rowlen = 0;         // halfs per plane row
  int ngroups_max = 0;
  Scratch u, v, work;
  CUtensorMap umap, vmap;
  explicit OzGemm(Pool* p) { u.pool = v.pool = work.pool = p; }
};

namespace {
// Stages per segment, segments per CTA and groups of a product over nstages
// stages and ntiles tiles: whole segments while the tiles fill the SMs, single
// stages per segment where the product is too small for that.
struct OzSplit {
  int seg, per, groups;
};
OzSplit oz_split(long long nstages, int ntiles, int nsm) {
  OzSplit s;
  s.seg = (int)std::max<long long>(1, std::min<long long>(oz64::kSegStages, nstages * ntiles / nsm));
  const long long nseg = (nstages + s.seg - 1) / s.seg;
  s.per = segs_per_cta(nseg, ntiles, nsm);
  s.groups = (int)((nseg + s.per - 1) / s.per);
  return s;
}

// Sizes of the planes (bytes) and partial sums for chunks of g->kpad inner
// values, the last of `last`.
struct OzBytes {
  size_t u, v, work;
  size_t total() const { return u + v + work; }
};
OzBytes oz_bytes(OzGemm* g, bool two, int ntiles, int nsm, long long last, bool real) {
  using namespace oz64;
  const long long spp = real ? SK : SK / 2;   // pairs per stage
  g->rowlen = (size_t)(g->kpad / spp) * SK;
  const int ga = oz_split(g->kpad / spp, ntiles, nsm).groups, gb = oz_split((last + spp - 1) / spp, ntiles, nsm).groups;
  g->ngroups_max = std::max(ga, gb);
  OzBytes b;
  b.u = (size_t)S * g->urows * g->rowlen * 2;
  b.v = two ? (size_t)S * g->vrows * g->rowlen * 2 : 0;
  b.work = (size_t)g->ngroups_max * ntiles * kTileElems * sizeof(double2);
  return b;
}

int oz_alloc(Ctx* c, OzGemm* g, bool two, int ntiles, int nsm, long long last, bool real) {
  const OzBytes b = oz_bytes(g, two, ntiles, nsm, last, real);
  if (b.total() > c->digit_room) return BGW_ENOMEM;
  int rc;
  if ((rc = c->pool.alloc(b.u, &g->u.ptr)) != BGW_OK) return rc;
  if (two && (rc = c->pool.alloc(b.v, &g->v.ptr)) != BGW_OK) return rc;
  return c->pool.alloc(b.work, &g->work.ptr);
}

void oz_release(Ctx* c, OzGemm* g) {
  for (Scratch* s : {&g->u, &g->v, &g->work}) {
    if (s->ptr) c->pool.release(s->ptr);
    s->ptr = nullptr;
  }
}

int oz_maps(Ctx* c, OzGemm* g) {
  using namespace oz64;
  TensorMapEncode enc;
  int rc = tensor_map_encode(c, &enc);
  if (rc != BGW_OK) return rc;
  for (int k = 0; k < 2; ++k) {
    void* base = k && g->v.ptr ? g->v.ptr : g->u.ptr;
    const int rows = k ? g->vrows : g->urows;
    cuuint64_t gdim[2] = {(cuuint64_t)g->rowlen, (cuuint64_t)S * rows};
    cuuint64_t gstride[1] = {(cuuint64_t)g->rowlen * 2};
    cuuint32_t box[2] = {(cuuint32_t)SK, (cuuint32_t)(k ? BN : BM)};
    cuuint32_t estr[2] = {1, 1};
    CUresult cr = enc(k ? &g->vmap : &g->umap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, base, gdim, gstride, box, estr,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (cr != CUDA_SUCCESS) return fail(c, BGW_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)cr);
  }
  return BGW_OK;
}

template <bool REALV>
int oz_launch(Ctx* c, const OzGemm& g, long long nstages, const OzSplit& s, int ntiles, const int2* tiles,
              const int* ufield, const int* vfield, const int* flag, cudaStream_t st) {
  using namespace oz64;
  BGW_CUDA(c, cudaFuncSetAttribute(gemm_kernel<REALV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
  gemm_kernel<REALV><<<(unsigned)((long long)s.groups * ntiles), kThreads, kSmem, st>>>(
      g.umap, g.vmap, g.urows, g.vrows, (int)nstages, s.seg, s.per, ntiles, tiles, ufield, vfield, flag, c->wait_ns,
      g.work.as<double2>(), c->d_status);
  BGW_CUDA(c, cudaGetLastError());
  c->launches += 1;
  return BGW_OK;
}
}  // namespace

namespace {
// Tiles of the product (lower ones alone for the Hermitian one).
std::vector<int2> oz_tiles(int ng, bool general) {
  using namespace oz64;
  const int nI = (ng + BM - 1) / BM, nJ = (ng + BN - 1) / BN;
  std::vector<int2> tl;
  for (int I = 0; I < nI; ++I)
    for (int J = 0; J < nJ; ++J)
      if (general || J * BN <= I * BM + BM - 1) tl.push_back(make_int2(I, J));
  return tl;
}

// Pairs per chunk: whole segments within kOzChunkBytes of digits.
long long oz_chunk(long long K, int rows, bool general, bool real) {
  using namespace oz64;
  const long long spp = real ? SK : SK / 2, whole = (K + spp - 1) / spp * spp;
  const long long seg_pairs = kSegStages * spp, per_pair = (long long)S * rows * (real ? 2 : 4) * (general ? 2 : 1);
  const long long kc = std::min<long long>((long long)(kOzChunkBytes / per_pair) / seg_pairs * seg_pairs, whole);
  return std::max<long long>(kc, std::min<long long>(seg_pairs, whole));
}
}  // namespace

size_t chi_oz_bytes(Ctx* c, long long K, int ng) {
  using namespace oz64;
  OzGemm g(&c->pool);
  g.urows = g.vrows = (ng + BM - 1) / BM * BM;
  const long long kc = oz_chunk(K, g.urows, false, false);
  g.kpad = kc;
  const size_t b = oz_bytes(&g, false, (int)oz_tiles(ng, false).size(), sm_count(c), K - (K - 1) / kc * kc, false).total();
  return b + (size_t(4) << 20);   // the pool rounds each block up to 2 MiB
}

// The FP64 polarizability of nrow frequencies on the tensor cores.  wr: real
// weights (Hermitian product; real: real M and chi), wc: complex weights (the
// real axis: every element).  *flags [nrow] (device, zeroed here): set where
// an operand is not finite or the pairs spread too far (kSpreadBits), the rows
// the caller's FMA kernel must do.
// *chunk: pairs per chunk as a run before took them, or 0 to size it here; the
// size taken is left there.  Returns BGW_ENOMEM when the scratch does not fit
// (nothing was launched).
int chi_oz_run(Ctx* c, long long K, int ng, const void* M, const double* wr, const double2* wc, int nrow, double scale,
               int accumulate, void* chi, bool real, int* flags, long long* chunk, cudaStream_t st) {
  using namespace oz64;
  const bool general = wc != nullptr;
  const int nsm = sm_count(c);
  const int rows = (ng + BM - 1) / BM * BM;
  const long long spp = real ? SK : SK / 2, seg_pairs = kSegStages * spp;
  const std::vector<int2> tl = oz_tiles(ng, general);
  const int ntiles = (int)tl.size();
  int rc;
  OzGemm g(&c->pool);
  Scratch meta, fac;
  meta.pool = fac.pool = &c->pool;
  // sizes of the operands (two where the columns' differ from the rows'), and the pairs' factors
  const int nop = general ? 2 : 1;
  const size_t meta_bytes = (size_t)nop * (rows + K + 1) * sizeof(int);
  g.urows = g.vrows = rows;
  long long kc = oz_chunk(K, rows, general, real);
  if (*chunk > 0) kc = *chunk;
  if ((rc = c->pool.alloc(meta_bytes, &meta.ptr)) != BGW_OK) return rc;
  if ((rc = c->pool.alloc((size_t)K * (general ? 3 : 1) * sizeof(double), &fac.ptr)) != BGW_OK) return rc;
  for (;;) {
    g.kpad = (kc + spp - 1) / spp * spp;
    const long long last = K - (K - 1) / kc * kc;
    rc = oz_alloc(c, &g, general, ntiles, nsm, last, real);
    if (rc == BGW_OK) break;
    oz_release(c, &g);
    if (kc <= kMinChunk || rc != BGW_ENOMEM) return rc;
    kc = std::max<long long>(kc / 2 / seg_pairs * seg_pairs, seg_pairs);
  }
  *chunk = kc;
  const void* d_tiles;
  if ((rc = upload_cached(c, tl.data(), tl.size() * sizeof(int2), st, &d_tiles)) != BGW_OK) return rc;
  const int2* tiles = static_cast<const int2*>(d_tiles);
  if ((rc = oz_maps(c, &g)) != BGW_OK) return rc;
  Sizes sz[2];
  for (int k = 0; k < nop; ++k) {
    sz[k].col = meta.as<int>() + (size_t)k * (rows + K + 1);
    sz[k].pair = sz[k].col + rows;
    sz[k].done = sz[k].pair + K;
  }
  const int *field = sz[0].col, *yfield = sz[nop - 1].col;
  double2* wf = general ? fac.as<double2>() : nullptr;   // 16-byte aligned: before the roots
  double* fp = general ? fac.as<double>() + 2 * K : fac.as<double>();
  BGW_CUDA(c, cudaMemsetAsync(flags, 0, nrow * sizeof(int), st));
  for (int f = 0; f < nrow; ++f) {
    int* flag = flags + f;
    {
      TimedScope ts(c, kTChiSplit, st);
      BGW_CUDA(c, cudaMemsetAsync(meta.ptr, 0, meta_bytes, st));
      sqrt_weights_kernel<<<(unsigned)((K + 255) / 256), 256, 0, st>>>(
          general ? nullptr : wr + (size_t)f * K, general ? wc + (size_t)f * K : nullptr, K, fp, wf);
      if (real)
        launch_colmax<kReal>(c, M, fp, nullptr, K, ng, sz[0], flag, st);
      else
        launch_colmax<kHerm>(c, M, fp, nullptr, K, ng, sz[0], flag, st);
      if (general) launch_colmax<kWeighted>(c, M, nullptr, wf, K, ng, sz[1], flag, st);
      c->launches += 1 + nop;
    }
    for (long long p0 = 0; p0 < K; p0 += kc) {
      const long long kn = std::min(kc, K - p0), nst = (kn + spp - 1) / spp;
      {
        TimedScope ts(c, kTChiSplit, st);
        const dim3 grid((unsigned)((nst * spp + 31) / 32), (unsigned)(rows / 32));
        // rows of the planes are rowlen long; a shorter last chunk fills the
        // first nst stages of each row and the product reads no further
        __half* up = g.u.as<__half>();
        if (real)
          digits_kernel<kReal><<<grid, 256, 0, st>>>(M, fp, nullptr, p0, kn, ng, rows, g.rowlen, field, flag, up);
        else
          digits_kernel<kHerm><<<grid, 256, 0, st>>>(M, fp, nullptr, p0, kn, ng, rows, g.rowlen, field, flag, up);
        if (general) {
          digits_kernel<kWeighted>
              <<<grid, 256, 0, st>>>(M, nullptr, wf, p0, kn, ng, rows, g.rowlen, yfield, flag, g.v.as<__half>());
          c->launches += 1;
        }
        BGW_CUDA(c, cudaGetLastError());
        c->launches += 1;
      }
      const OzSplit s = oz_split(nst, ntiles, nsm);
      {
        TimedScope ts(c, kTChiTc, st);
        rc = real ? oz_launch<true>(c, g, nst, s, ntiles, tiles, field, yfield, flag, st)
                  : oz_launch<false>(c, g, nst, s, ntiles, tiles, field, yfield, flag, st);
        if (rc != BGW_OK) return rc;
      }
      {
        TimedScope ts(c, kTChiReduce, st);
        const unsigned nb = (unsigned)(((long long)ntiles * kTileElems + 255) / 256);
        const int acc = accumulate || p0 > 0;
        if (real)
          reduce_kernel<true, true><<<nb, 256, 0, st>>>(g.work.as<double2>(), s.groups, ntiles, tiles, ng, -scale, acc,
                                                        flag, static_cast<double*>(chi) + (size_t)f * ng * ng);
        else if (general)
          reduce_kernel<false, false><<<nb, 256, 0, st>>>(g.work.as<double2>(), s.groups, ntiles, tiles, ng, scale,
                                                          acc, flag, static_cast<double2*>(chi) + (size_t)f * ng * ng);
        else
          reduce_kernel<true, false><<<nb, 256, 0, st>>>(g.work.as<double2>(), s.groups, ntiles, tiles, ng, -scale,
                                                         acc, flag, static_cast<double2*>(chi) + (size_t)f * ng * ng);
        BGW_CUDA(c, cudaGetLastError());
        c->launches += 1;
      }
    }
  }
  return BGW_OK;
}

// The FP64 Sigma forms qW_p = m_p^H W m_p and qV_p = sum_G |m_p(G)|^2 v_G of K
// pairs on the tensor cores: C = W m by digit products (rows of conj(m) against
// rows of W, inner index G'), block by block of pairs.  *flag (device, zeroed
// here) is set where an operand is not finite: the FMA kernels must then do the
// call.  Returns BGW_ENOMEM when the scratch does not fit (nothing launched).
int sigma_oz_forms(Ctx* c, long long K, int ng, const void* M, const void* W, const double* sv, double* qW, double* qV,
                   int* flag, cudaStream_t st) {
  using namespace oz64;
  const int nsm = sm_count(c);
  const int nJ = (ng + BN - 1) / BN;
  const long long nst = (ng + SK / 2 - 1) / (SK / 2);
  OzGemm g(&c->pool);
  g.kpad = nst * (SK / 2);
  g.vrows = nJ * BN;
  Scratch meta;
  meta.pool = &c->pool;
  const size_t row_bytes = (size_t)S * g.kpad * 2 * 2;
  long long rows = std::min<long long>((K + BM - 1) / BM * BM,
                                       std::max<long long>(BM, (long long)(kOzChunkBytes / 2 / row_bytes) / BM * BM));
  int rc;
  if ((rc = c->pool.alloc((size_t)(rows + g.vrows) * sizeof(int), &meta.ptr)) != BGW_OK) return rc;
  for (;;) {
    g.urows = (int)rows;
    rc = oz_alloc(c, &g, true, (int)(rows / BM) * nJ, nsm, g.kpad, false);
    if (rc == BGW_OK) break;
    oz_release(c, &g);
    if (rc != BGW_ENOMEM || rows == BM) return rc;
    rows = std::max<long long>(BM, rows / 2 / BM * BM);
  }
  std::vector<int2> tl;
  for (int I = 0; I < (int)(rows / BM); ++I)
    for (int J = 0; J < nJ; ++J) tl.push_back(make_int2(I, J));
  const void* d_tiles;
  if ((rc = upload_cached(c, tl.data(), tl.size() * sizeof(int2), st, &d_tiles)) != BGW_OK) return rc;
  if ((rc = oz_maps(c, &g)) != BGW_OK) return rc;
  int* ufield = meta.as<int>();
  int* vfield = ufield + rows;
  BGW_CUDA(c, cudaMemsetAsync(flag, 0, sizeof(int), st));
  row_digits_kernel<<<(g.vrows + 7) / 8, 256, 0, st>>>(static_cast<const double2*>(W), ng, ng, g.vrows, g.rowlen, 0,
                                                       vfield, flag, g.v.as<__half>());
  for (long long p0 = 0; p0 < K; p0 += rows) {
    const int R = (int)std::min<long long>(rows, K - p0), nI = (R + BM - 1) / BM, ntiles = nI * nJ;
    row_digits_kernel<<<nI * BM / 8, 256, 0, st>>>(static_cast<const double2*>(M) + (size_t)p0 * ng, R, ng, g.urows,
                                                   g.rowlen, 1, ufield, flag, g.u.as<__half>());
    BGW_CUDA(c, cudaGetLastError());
    OzSplit s = oz_split(nst, ntiles, nsm);
    s.groups = std::min(s.groups, g.ngroups_max * (int)(rows / BM) * nJ / ntiles);   // fits the partial sums' space
    s.per = (int)((((nst + s.seg - 1) / s.seg) + s.groups - 1) / s.groups);
    if ((rc = oz_launch<false>(c, g, nst, s, ntiles, static_cast<const int2*>(d_tiles), ufield, vfield, flag, st)) !=
        BGW_OK)
      return rc;
    sigma_forms_kernel<<<(R + 7) / 8, 256, 0, st>>>(static_cast<const double2*>(M), p0, R, ng, sv,
                                                    g.work.as<double2>(), s.groups, ntiles, flag, qW, qV);
    BGW_CUDA(c, cudaGetLastError());
    c->launches += 2;
  }
  c->launches += 1;
  return BGW_OK;
}

}  // namespace bgw
