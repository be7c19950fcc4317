// General (non-Hermitian) dielectric matrix and its inverse, for the real-axis
// response of Eq. retarded_advanced_epsilon: with complex pair weights chi is
// no longer Hermitian, eps~ = I - V^1/2 chi V^1/2 is a general complex matrix,
// and its inverse needs pivoting (the paper inverts with ZGESV, an LU with
// partial pivoting).
//
// Blocked Gauss-Jordan elimination with row interchanges, 32 columns a step:
//   1. pivot rows for the block's columns among the rows not yet used, chosen
//      by tournament pivoting: CTAs run a partial-pivoting LU on 256-row
//      slices of the column panel and keep 32 candidates each; merge rounds
//      run the same LU on up to 8 candidate sets at a time until 32 rows
//      remain (the selection of a partial-pivoting LU of the panel when one
//      slice holds every row, a tournament among slices otherwise).  The
//      selection LUs run in FP32: they only choose rows;
//   2. the chosen rows are swapped into the block's rows (whole rows of the
//      working matrix: row operations on the augmented system), the
//      interchanges recorded LAPACK-style (ipiv[j] >= j);
//   3. one Gauss-Jordan block step without further pivoting (the block's
//      diagonal block is the chosen rows, eliminated in their selection order).
// After the last step the working matrix holds the inverse with permuted
// columns; undoing the interchanges on the columns in reverse order gives
// eps~^-1.
#include <algorithm>
#include <memory>
#include <vector>

#include "runtime.h"
#include "sweep_common.cuh"

namespace bgw {

namespace {

constexpr int kPB = 32;      // block width of the Gauss-Jordan step
constexpr int kTRows = 256;  // rows per selection CTA (one per thread)
constexpr int kSwapCols = 64;
constexpr int kGB = 16;      // matrices of one size stepped together (grid.y / grid.z = matrix)

struct GenPtrs {
  double2* A[kGB];
};

// z + a b
__device__ __forceinline__ double2 cfma2(double2 a, double2 b, double2 z) {
  z.x = fma(a.x, b.x, z.x);
  z.y = fma(a.x, b.y, z.y);
  z.x = fma(-a.y, b.y, z.x);
  z.y = fma(a.y, b.x, z.y);
  return z;
}

__device__ __forceinline__ double2 cmul2(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}

// z - a b, four FP64 FMAs
__device__ __forceinline__ double2 cfnma2(double2 a, double2 b, double2 z) {
  z.x = fma(-a.x, b.x, z.x);
  z.y = fma(-a.x, b.y, z.y);
  z.x = fma(a.y, b.y, z.x);
  z.y = fma(-a.y, b.x, z.y);
  return z;
}

// z - a b with one rounding of z
__device__ __forceinline__ double2 csub2(double2 z, double2 a, double2 b) {
  const double2 t = cmul2(a, b);
  return make_double2(z.x - t.x, z.y - t.y);
}

__device__ __forceinline__ double2 shfl2(double2 v, int src, int width = 32) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, src, width), __shfl_sync(0xffffffffu, v.y, src, width));
}

// FP32 copy of a panel entry, rounded in the integer pipe (a conversion goes
// through the FP64 pipe: 4 us of a CTA's 16384).  The values are eps~ entries
// (finite, far inside the FP32 range); a zero pivot column stays zero.
__device__ __forceinline__ float2 to_f2(double2 z) { return make_float2(ff_from_int(z.x).x, ff_from_int(z.y).x); }

// Partial-pivoting LU of nr (<= 256) rows gid[] x kb columns of the panel at
// column k0; thread t owns row t and keeps it in registers.  Picks, column by
// column, the active row of largest |Re|+|Im| (ties: smallest global row),
// eliminates that column from the other active rows.  Writes the global rows
// in selection order to sel and returns their number (min(nr, kb)).  The
// selection runs in FP32: it only orders the rows (the elimination itself is
// the FP64 Gauss-Jordan step that follows), and FP32 runs at 64 times the
// FP64 rate of one SM.
//
// A chain of kb dependent searches bounds it.  Each warp finds its own best
// row with two redux instructions and lays that row down beside the key
// before the one barrier of the column; after it every warp compares the
// eight keys itself and reads the winner's row (two sets of rows, so the next
// column may write while this one is read).  About 33 us a launch once the rows
// are in L2, latencies of 32 columns with two warps a scheduler.
struct SelectSmem {
  float4 row[2][kTRows / 32][kPB / 2];
  uint2 key[2][kTRows / 32];   // (|Re|+|Im| as ordered bits + 1, global row); 0: no active row
};

// Columns [j0, j0 + 8) of the panel and the ones after them; x[0] is column j0
// of the thread's row.  The row moves down by one register with every column's
// update, so that the loop needs one body a stage: 32 unrolled columns are code
// that runs once, and with its fetches a launch took 50 us.
template <int J0>
__device__ __forceinline__ void select_stage(float2 (&x)[kPB], bool active, unsigned g, int cnt, SelectSmem& sm,
                                             int* sel) {
  constexpr int W = kPB - J0;   // columns left
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 1
  for (int j = J0; j < min(J0 + 8, cnt); ++j) {
    const float v = fabsf(x[0].x) + fabsf(x[0].y);
    const unsigned key = active ? (v == v ? __float_as_uint(v) : 0u) + 1u : 0u;
    const unsigned kmax = __reduce_max_sync(0xffffffffu, key);
    const unsigned gmin = __reduce_min_sync(0xffffffffu, key == kmax ? g : 0xffffffffu);
    if (kmax == 0 ? lane == 0 : (active && g == gmin)) {
      sm.key[j & 1][warp] = make_uint2(kmax, gmin);
#pragma unroll
      for (int c = 0; c < W / 2; ++c)
        sm.row[j & 1][warp][c] = make_float4(x[2 * c].x, x[2 * c].y, x[2 * c + 1].x, x[2 * c + 1].y);
    }
    __syncthreads();
    // the best of the eight: every warp by itself, lane = warp of the key
    const uint2 k = sm.key[j & 1][lane & 7];
    uint2 best;
    best.x = __reduce_max_sync(0xffffffffu, k.x);
    best.y = __reduce_min_sync(0xffffffffu, k.x == best.x ? k.y : 0xffffffffu);
    const int bw = __ffs(__ballot_sync(0xffffffffu, k.x == best.x && k.y == best.y)) - 1;
    if (threadIdx.x == 0) sel[j] = (int)best.y;
    if (g == best.y) active = false;
    const float4* row = sm.row[j & 1][bw];
    float4 q = row[0];
    const float m2 = q.x * q.x + q.y * q.y;
    float2 l = make_float2(0.f, 0.f);
    if (active && m2 > 0.f)
      l = make_float2((x[0].x * q.x + x[0].y * q.y) / m2, (x[0].y * q.x - x[0].x * q.y) / m2);
    auto sub = [&](float2 z, float ux, float uy) {
      return make_float2(fmaf(-l.x, ux, fmaf(l.y, uy, z.x)), fmaf(-l.x, uy, fmaf(-l.y, ux, z.y)));
    };
    if (active) {
      x[0] = sub(x[1], q.z, q.w);
#pragma unroll
      for (int c = 1; c < W / 2; ++c) {
        q = row[c];
        x[2 * c - 1] = sub(x[2 * c], q.x, q.y);
        x[2 * c] = sub(x[2 * c + 1], q.z, q.w);
      }
      x[W - 1] = make_float2(0.f, 0.f);
    }
  }
  if constexpr (J0 + 8 < kPB) select_stage<J0 + 8>(x, active, g, cnt, sm, sel);
}

__device__ __forceinline__ int select_rows(const double2* __restrict__ A, int ng, int k0, const int* gid, int nr,
                                           int kb, float2 (*P)[kPB + 1], SelectSmem& sm, int* sel) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  // coalesced: a warp reads its 32 rows, one row a load
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    const int r = 32 * warp + i;
    P[r][lane] = (r < nr && lane < kb) ? to_f2(A[(size_t)gid[r] * ng + k0 + lane]) : make_float2(0.f, 0.f);
  }
  __syncwarp();
  float2 x[kPB];
#pragma unroll
  for (int c = 0; c < kPB; ++c) x[c] = P[t][c];
  const int cnt = min(nr, kb);
  select_stage<0>(x, t < nr, t < nr ? (unsigned)gid[t] : 0xffffffffu, cnt, sm, sel);
  __syncthreads();
  return cnt;
}

// The CTA that makes the final choice leaves the block D = A[sel][K] (the
// chosen rows in selection order, identity outside kb) before the rows are
// swapped; the swap launch factors it beside the swaps.
__device__ __forceinline__ void stash_block(const double2* __restrict__ A, int ng, int k0, int kb, const int* sel,
                                            double2* __restrict__ lu) {
  for (int e = threadIdx.x; e < kPB * kPB; e += blockDim.x) {
    const int r = e / kPB, c = e % kPB;
    lu[e] = (r < kb && c < kb) ? A[(size_t)sel[r] * ng + k0 + c] : make_double2(r == c ? 1.0 : 0.0, 0.0);
  }
}

// FP64 LU (without further pivoting) of the stashed block, 256 threads: lu
// comes in as D[r][c] and goes out by columns, lu[c * NB + r] = L below the
// diagonal (unit diagonal implied) and U on and above it, lu[NB*NB + s] =
// 1/U_ss.  Lane = row, warp w holds columns w, w + 8, ... in registers; the
// row of U comes by shuffle, the column of L through shared memory, written
// for the next column by its warp ahead of that warp's other columns (one
// barrier a column).  41 us, bounded by that chain (its FP64 operations queue
// behind the other warps') and by the pipe (17 us with idle lanes); it runs
// beside the swaps (about 10 us).  With each product rounded apart from its
// element, 50 us; the inverse's error is below the older kernels' either way
// (by 2 to 30 % at N_G 37 to 900).
__device__ void factor_block(double2* __restrict__ lu, int kb, double2 (*Lb)[kPB], int* __restrict__ status) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double2 x[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) x[i] = lu[lane * kPB + warp + 8 * i];
  auto scale = [&](double2& v, int s) {   // column s: reciprocal pivot, L below it
    const double2 p = shfl2(v, s);
    const double m2 = p.x * p.x + p.y * p.y;
    const double q = rcp_f64_checked(m2, status);   // the same in every lane; 0 sets the status
    const double2 ri = make_double2(p.x * q, -p.y * q);
    if (lane > s) v = cmul2(v, ri);
    Lb[s & 1][lane] = v;
    if (lane == 0) lu[kPB * kPB + s] = ri;
  };
  __syncthreads();   // every element read before any is written back
  if (warp == 0) scale(x[0], 0);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    for (int q = 0; q < 8; ++q) {
      const int s = 8 * i + q;
      if (s >= kb) break;
      __syncthreads();
      const double2 l = Lb[s & 1][lane];
      auto upd = [&](double2& v) {
        const double2 u = shfl2(v, s);
        if (lane > s) v = cfnma2(l, u, v);
      };
      if (q < 7) {
        if (warp == q + 1 && s + 1 < kb) {
          upd(x[i]);
          scale(x[i], s + 1);
        } else if (warp > q) {
          upd(x[i]);
        }
        if (i < 3) upd(x[i < 3 ? i + 1 : 3]);
      } else if (i < 3) {
        upd(x[i < 3 ? i + 1 : 3]);
        if (warp == 0 && s + 1 < kb) scale(x[i < 3 ? i + 1 : 3], s + 1);
      }
#pragma unroll
      for (int h = 2; h < 4; ++h)
        if (i + h < 4) upd(x[i + h < 4 ? i + h : 3]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) lu[(warp + 8 * i) * kPB + lane] = x[i];
  if (threadIdx.x >= kb && threadIdx.x < kPB) lu[kPB * kPB + threadIdx.x] = make_double2(1.0, 0.0);
}

// Row panel R = D^-1 A_K,: from the factors (after the swap, row k0 + r is
// the r-th chosen row): L U x = b for every column of A_K,:, the block's own
// columns replaced by identity columns (R = D^-1 there).  CTAs after the
// first ceil(ng / 16) copy the column panel Cp = A_:,K (ld NB).
//
// The FP64 pipe (two FMAs a clock and SM) bounds it: 4600 operations a column.
// Four lanes hold a column, rows l, l + 4, ... in registers, so the chain needs
// shuffles and no barrier, and the triangles leave few lanes idle.  A row takes
// four solved rows at a time and rounds once for them: with one FMA after the
// other on the row itself the step takes 88 us but the inverse's error is 6 %
// larger than with a product rounded apart from the row, this way 5 % smaller.
// Five matrices of N_G 1643: 106 us a step (the FP64 pipe 88 % busy, 60 us of it
// the operations without the idle lanes and the last wave),
// CTAs of one warp for the last wave's sake (of two: 17 us more); 209 us with
// 16 columns by 16 row groups, shared memory and three barriers a row pair.
// SIZES (FP64 inputs): sizes[m][0 / 1][k], the largest exponent fields of
// row k of R and of column k of Cp outside the block's rows.
constexpr int kCopyRows = 32;
constexpr int kSolveThreads = 32, kSolveCols = kSolveThreads / 4;

template <bool SIZES>
__global__ void __launch_bounds__(kSolveThreads) solve_panels_kernel(const __grid_constant__ GenPtrs P, int ng,
                                                                     int k0, int kb,
                                                                     const double2* __restrict__ lu_all,
                                                                     double2* __restrict__ R_all,
                                                                     double2* __restrict__ C_all,
                                                                     int* __restrict__ sizes) {
  const int tid = threadIdx.x;
  const int m = blockIdx.y;
  const double2* __restrict__ A = P.A[m];
  const double2* __restrict__ lu = lu_all + (size_t)m * kPB * (kPB + 1);
  double2* __restrict__ R = R_all + (size_t)m * kPB * ng;
  double2* __restrict__ C = C_all + (size_t)m * kPB * ng;
  const int ncol = (ng + kSolveCols - 1) / kSolveCols;
  if ((int)blockIdx.x >= ncol) {   // kCopyRows rows of the column panel
    const int r0 = (blockIdx.x - ncol) * kCopyRows, s = tid & 31;
    int top = 0;
#pragma unroll 8
    for (int r = tid >> 5; r < kCopyRows; r += kSolveThreads / 32)
      if (s < kb && r0 + r < ng) {
        const double2 v = A[(size_t)(r0 + r) * ng + k0 + s];
        C[(size_t)(r0 + r) * kPB + s] = v;
        if (SIZES && (r0 + r < k0 || r0 + r >= k0 + kb)) top = max(top, max(exponent_field(v.x), exponent_field(v.y)));
      }
    if (SIZES && top) atomicMax(sizes + (m * 2 + 1) * kPB + s, top);
    return;
  }
  __shared__ double2 D[kPB][kPB];   // by columns
  __shared__ double2 rinv[kPB];
  const int l = tid & 3;
  const int j = blockIdx.x * kSolveCols + (tid >> 2);
  double2 x[8];
#pragma unroll
  for (int h = 0; h < 8; ++h) {
    const int r = l + 4 * h;
    x[h] = make_double2(0.0, 0.0);
    if (r < kb && j < ng)
      x[h] = (j >= k0 && j < k0 + kb) ? make_double2(j - k0 == r ? 1.0 : 0.0, 0.0) : A[(size_t)(k0 + r) * ng + j];
  }
#pragma unroll 8
  for (int e = tid; e < kPB * kPB; e += kSolveThreads) (&D[0][0])[e] = lu[e];
  if (tid < kPB) rinv[tid] = lu[kPB * kPB + tid];
  __syncthreads();
  // rows 4 i + l take four solved rows 4 h .. 4 h + 3 at a time, their sum rounded to x once
  auto rest = [&](double2& xi, int h, int i, const double2 (&y)[4]) {
    double2 t = cmul2(D[4 * h][l + 4 * i], y[0]);
#pragma unroll
    for (int q = 1; q < 4; ++q) t = cfma2(D[4 * h + q][l + 4 * i], y[q], t);
    xi = make_double2(xi.x - t.x, xi.y - t.y);
  };
  double2 y[4];
#pragma unroll
  for (int h = 0; h < 8; ++h) {   // unit lower factor
    if (4 * h >= kb) break;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      y[q] = shfl2(x[h], q, 4);
      if (l > q) x[h] = csub2(x[h], D[4 * h + q][l + 4 * h], y[q]);
    }
#pragma unroll
    for (int i = h + 1; i < 8; ++i) rest(x[i], h, i, y);
  }
#pragma unroll
  for (int h = 7; h >= 0; --h) {   // upper factor
    if (4 * h >= kb) continue;
#pragma unroll
    for (int q = 3; q >= 0; --q) {
      if (l == q) x[h] = cmul2(x[h], rinv[4 * h + q]);
      y[q] = shfl2(x[h], q, 4);
      if (l < q) x[h] = csub2(x[h], D[4 * h + q][l + 4 * h], y[q]);
    }
#pragma unroll
    for (int i = h - 1; i >= 0; --i) rest(x[i], h, i, y);
  }
#pragma unroll
  for (int h = 0; h < 8; ++h) {
    const int r = l + 4 * h;
    if (r < kb && j < ng) R[(size_t)r * ng + j] = x[h];
  }
  if constexpr (!SIZES) return;
#pragma unroll
  for (int h = 0; h < 8; ++h) {   // largest of the warp's columns in rows l + 4 h
    int top = max(exponent_field(x[h].x), exponent_field(x[h].y));
    for (int o = 4; o < 32; o <<= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    if (tid < 4 && top) atomicMax(sizes + m * 2 * kPB + l + 4 * h, top);
  }
}

// Leaf round: CTA b takes rows k0 + 256 b ... of the panel.
__global__ void __launch_bounds__(kTRows) pivot_leaf_kernel(const __grid_constant__ GenPtrs Pm, int ng, int k0,
                                                            int kb, int* __restrict__ out_all, int cstride,
                                                            double2* __restrict__ lu_all) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int m = blockIdx.y;
  const double2* __restrict__ A = Pm.A[m];
  int* __restrict__ out = out_all + (size_t)m * cstride;
  int* __restrict__ cnt = out + (cstride / (kPB + 1)) * kPB;
  double2* __restrict__ lu = lu_all + (size_t)m * kPB * (kPB + 1);
  float2 (*P)[kPB + 1] = reinterpret_cast<float2 (*)[kPB + 1]>(smem_raw);
  __shared__ int gid[kTRows];
  __shared__ int sel[kPB];
  __shared__ SelectSmem sm;
  const int r0 = k0 + blockIdx.x * kTRows;
  const int nr = min(kTRows, ng - r0);
  const int t = threadIdx.x;
  gid[t] = r0 + t;
  __syncthreads();
  const int n = select_rows(A, ng, k0, gid, nr, kb, P, sm, sel);
  if (t < n) out[blockIdx.x * kPB + t] = sel[t];
  if (t == 0) cnt[blockIdx.x] = n;
  if (gridDim.x == 1) stash_block(A, ng, k0, kb, sel, lu);   // the final choice
}

// Merge round: CTA m takes candidate sets 8m .. 8m+7 (of ngroups).
__global__ void __launch_bounds__(kTRows) pivot_merge_kernel(const __grid_constant__ GenPtrs Pm, int ng, int k0,
                                                             int kb, const int* __restrict__ in_all,
                                                             int ngroups, int* __restrict__ out_all, int cstride,
                                                             double2* __restrict__ lu_all) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int m = blockIdx.y;
  const double2* __restrict__ A = Pm.A[m];
  const int* __restrict__ in = in_all + (size_t)m * cstride;
  const int* __restrict__ cin = in + (cstride / (kPB + 1)) * kPB;
  int* __restrict__ out = out_all + (size_t)m * cstride;
  int* __restrict__ cout = out + (cstride / (kPB + 1)) * kPB;
  double2* __restrict__ lu = lu_all + (size_t)m * kPB * (kPB + 1);
  float2 (*P)[kPB + 1] = reinterpret_cast<float2 (*)[kPB + 1]>(smem_raw);
  __shared__ int gid[kTRows];
  __shared__ int sel[kPB];
  __shared__ SelectSmem sm;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int g0 = blockIdx.x * 8;
  int before = 0, nr = 0, mine = 0;   // rows of the sets before this warp's, of all, of its own
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = g0 + i < ngroups ? cin[g0 + i] : 0;
    if (i < warp) before += k;
    if (i == warp) mine = k;
    nr += k;
  }
  if (lane < mine) gid[before + lane] = in[(g0 + warp) * kPB + lane];
  __syncthreads();
  const int n = select_rows(A, ng, k0, gid, nr, kb, P, sm, sel);
  if (t < n) out[blockIdx.x * kPB + t] = sel[t];
  if (t == 0) cout[blockIdx.x] = n;
  if (gridDim.x == 1) stash_block(A, ng, k0, kb, sel, lu);   // the final choice
}

// Brings row sel[j] to row k0 + j for j < kb by successive interchanges
// (recorded in ipiv[k0 + j]).  Every CTA but the last replays the
// interchanges on the set of affected rows (at most 64; one warp, two slots a
// lane) and moves its 64 columns of them.  The last CTA factors the stashed
// block meanwhile.
__global__ void __launch_bounds__(256) pivot_swap_kernel(const __grid_constant__ GenPtrs Pm, int ng, int k0, int kb,
                                                         const int* __restrict__ sel_all, int cstride,
                                                         int* __restrict__ ipiv_all, double2* __restrict__ lu_all,
                                                         int* __restrict__ sizes, int* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int m = blockIdx.y;
  if (blockIdx.x == gridDim.x - 1) {
    if (sizes && threadIdx.x < 2 * kPB) sizes[m * 2 * kPB + threadIdx.x] = 0;   // solve_panels_kernel fills them
    factor_block(lu_all + (size_t)m * kPB * (kPB + 1), kb, reinterpret_cast<double2 (*)[kPB]>(smem_raw), status);
    return;
  }
  double2* __restrict__ A = Pm.A[m];
  const int* __restrict__ sel = sel_all + (size_t)m * cstride;
  int* __restrict__ ipiv = ipiv_all + (size_t)m * ng;
  double2 (*buf)[kSwapCols] = reinterpret_cast<double2 (*)[kSwapCols]>(smem_raw);
  __shared__ int pos[2 * kPB];   // positions of the affected rows (-1: none)
  __shared__ int from[2 * kPB];  // original row that ends at pos[i]
  const int t = threadIdx.x;
  if (t < 32) {
    const int sj = t < kb ? sel[t] : -1;
    const bool far = sj >= k0 + kb;   // a row outside the block's own
    const unsigned fm = __ballot_sync(0xffffffffu, far);
    pos[t] = t < kb ? k0 + t : -1;
    pos[kPB + t] = -1;
    __syncwarp();
    if (far) pos[kPB + __popc(fm & ((1u << t) - 1))] = sj;
    __syncwarp();
    int f0 = pos[t], f1 = pos[kPB + t];
    for (int j = 0; j < kb; ++j) {
      const int want = __shfl_sync(0xffffffffu, sj, j);
      const int old = __shfl_sync(0xffffffffu, f0, j);
      const unsigned b0 = __ballot_sync(0xffffffffu, f0 == want), b1 = __ballot_sync(0xffffffffu, f1 == want);
      const int cur = b0 ? __ffs(b0) - 1 : kPB + __ffs(b1) - 1;   // slot holding original row sel[j]
      if (t == j) f0 = want;
      if (cur < kPB) {
        if (t == cur) f0 = old;
      } else if (t == cur - kPB) {
        f1 = old;
      }
      if (blockIdx.x == 0 && t == 0) ipiv[k0 + j] = pos[cur];
    }
    from[t] = f0;
    from[kPB + t] = f1;
  }
  __syncthreads();
  const int c0 = blockIdx.x * kSwapCols;
#pragma unroll 8
  for (int e = t; e < 2 * kPB * kSwapCols; e += 256) {
    const int i = e / kSwapCols, cc = e % kSwapCols;
    if (c0 + cc < ng && from[i] != pos[i]) buf[i][cc] = A[(size_t)from[i] * ng + c0 + cc];
  }
  __syncthreads();
#pragma unroll 8
  for (int e = t; e < 2 * kPB * kSwapCols; e += 256) {
    const int i = e / kSwapCols, cc = e % kSwapCols;
    if (c0 + cc < ng && from[i] != pos[i]) A[(size_t)pos[i] * ng + c0 + cc] = buf[i][cc];
  }
}

// Column j of the inverse is column src[j] of the working matrix: the
// interchanges undone on the columns, last first.
// The chain of interchanges runs in shared memory.
__global__ void __launch_bounds__(256) colperm_build_kernel(const int* __restrict__ ipiv_all, int ng,
                                                            int* __restrict__ src_all) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int* src = reinterpret_cast<int*>(smem_raw);
  int* ipiv = src + ng;
  for (int j = threadIdx.x; j < ng; j += 256) {
    src[j] = j;
    ipiv[j] = ipiv_all[(size_t)blockIdx.x * ng + j];
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int j = ng - 1; j >= 0; --j) {
      const int p = ipiv[j];
      const int tmp = src[j];
      src[j] = src[p];
      src[p] = tmp;
    }
  __syncthreads();
  for (int j = threadIdx.x; j < ng; j += 256) src_all[(size_t)blockIdx.x * ng + j] = src[j];
}

__global__ void __launch_bounds__(256) colperm_apply_kernel(const __grid_constant__ GenPtrs Pm, int ng,
                                                            const int* __restrict__ src_all) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* row = reinterpret_cast<double2*>(smem_raw);
  double2* a = Pm.A[blockIdx.y] + (size_t)blockIdx.x * ng;
  const int* __restrict__ src = src_all + (size_t)blockIdx.y * ng;
  for (int j = threadIdx.x; j < ng; j += 256) row[j] = a[j];
  __syncthreads();
  for (int j = threadIdx.x; j < ng; j += 256) a[j] = row[src[j]];
}

}  // namespace

int epsinv_general_run(Ctx* c, int nmat, const int* ng, const bgw_cell* const* cells, const int32_t* const* d_geps,
                       const void* const* chi, void* const* eps, void* const* epsinv, cudaStream_t st,
                       bool tc_update) {
  int ngmax = 0;
  for (int m = 0; m < nmat; ++m) ngmax = std::max(ngmax, ng[m]);
  const int nleaf_max = (ngmax + kTRows - 1) / kTRows;
  const int cstride = nleaf_max * (kPB + 1);   // candidates then counts, per matrix
  Scratch sv, lu, R, Cp, cand, ipiv;
  sv.pool = lu.pool = R.pool = Cp.pool = cand.pool = ipiv.pool = &c->pool;
  const size_t lu_bytes = (size_t)kGB * kPB * (kPB + 1) * sizeof(double2);   // the operands' sizes follow
  int rc;
  if ((rc = c->pool.alloc((size_t)ngmax * sizeof(double), &sv.ptr)) != BGW_OK ||
      (rc = c->pool.alloc(lu_bytes + (size_t)kGB * 2 * kPB * sizeof(int), &lu.ptr)) != BGW_OK ||
      (rc = c->pool.alloc((size_t)kGB * kPB * ngmax * sizeof(double2), &R.ptr)) != BGW_OK ||
      (rc = c->pool.alloc((size_t)kGB * kPB * ngmax * sizeof(double2), &Cp.ptr)) != BGW_OK ||
      (rc = c->pool.alloc((size_t)2 * kGB * cstride * sizeof(int), &cand.ptr)) != BGW_OK ||
      (rc = c->pool.alloc((size_t)2 * kGB * ngmax * sizeof(int), &ipiv.ptr)) != BGW_OK)
    return fail(c, rc, "general inverse: scratch allocation failed");
  const size_t psmem = sizeof(float2) * kTRows * (kPB + 1);
  const size_t ssmem = sizeof(double2) * 2 * kPB * kSwapCols;
  BGW_CUDA(c, allow_smem(reinterpret_cast<const void*>(pivot_leaf_kernel), psmem));
  BGW_CUDA(c, allow_smem(reinterpret_cast<const void*>(pivot_merge_kernel), psmem));
  BGW_CUDA(c, allow_smem(reinterpret_cast<const void*>(pivot_swap_kernel), ssmem));
  BGW_CUDA(c, allow_smem(reinterpret_cast<const void*>(colperm_build_kernel), 2 * sizeof(int) * ngmax));
  BGW_CUDA(c, allow_smem(reinterpret_cast<const void*>(colperm_apply_kernel), sizeof(double2) * ngmax));
  int* cbuf[2] = {cand.as<int>(), cand.as<int>() + (size_t)kGB * cstride};
  // Matrices of equal size are stepped together, up to kGB at a time: every
  // launch below serves the whole group.
  for (int m0 = 0; m0 < nmat;) {
    const int n = ng[m0];
    int nb = 1;
    while (m0 + nb < nmat && nb < kGB && ng[m0 + nb] == n) ++nb;
    GenPtrs P = {};
    for (int k = 0; k < nb; ++k) {
      const int m = m0 + k;
      P.A[k] = static_cast<double2*>(epsinv[m]);
      if ((rc = eps_form_run(c, cells[m], d_geps[m], n, chi[m], sv.as<double>(), P.A[k], eps ? eps[m] : nullptr,
                             st)) != BGW_OK)
        return rc;
    }
    TimedScope ts(c, kTInverse, st);
    std::unique_ptr<OzPlan, void (*)(OzPlan*)> oz(nullptr, oz_plan_delete);
    long long way = -1;   // sets of slices; 0: the FMA sweep
    if (tc_update) c->routes.given(&way);
    if (tc_update && way != 0) {
      oz.reset(oz_plan_new());
      std::vector<int> ngs(nb, n);
      std::vector<double2*> As(nb);
      std::vector<const double2*> Rs(nb), Cs(nb);
      for (int k = 0; k < nb; ++k) {
        As[k] = P.A[k];
        Rs[k] = R.as<double2>() + (size_t)k * kPB * n;
        Cs[k] = Cp.as<double2>() + (size_t)k * kPB * n;
      }
      rc = oz_prepare(c, nb, ngs.data(), As.data(), Rs.data(), Cs.data(), nullptr, oz.get(), true, false,
                      c->run_slices, c->run_ff_chain, (int)way);
      if (fma_fallback(c, rc))
        oz.reset();
      else if (rc != BGW_OK)
        return rc;
      else
        oz_set_bulk_items(oz.get(), c->update_items);   // the option's width, else the SM-count rule
      c->routes.note(oz ? oz_buffers(oz.get()) : 0);
    }
    int* sizes = oz && !c->run_ff_chain ? reinterpret_cast<int*>(static_cast<char*>(lu.ptr) + lu_bytes) : nullptr;
    int* piv = ipiv.as<int>();
    int* src = piv + (size_t)kGB * ngmax;
    for (int k0 = 0; k0 < n; k0 += kPB) {
      const int kb = std::min(kPB, n - k0);
      int groups = (n - k0 + kTRows - 1) / kTRows;
      int cur = 0;
      {
        TimedScope tp(c, kTPivot, st);
        pivot_leaf_kernel<<<dim3(groups, nb), kTRows, psmem, st>>>(P, n, k0, kb, cbuf[0], cstride, lu.as<double2>());
        c->launches += 1;
        while (groups > 1) {
          const int next = (groups + 7) / 8;
          pivot_merge_kernel<<<dim3(next, nb), kTRows, psmem, st>>>(P, n, k0, kb, cbuf[cur], groups, cbuf[1 - cur],
                                                                    cstride, lu.as<double2>());
          c->launches += 1;
          cur = 1 - cur;
          groups = next;
        }
        pivot_swap_kernel<<<dim3((n + kSwapCols - 1) / kSwapCols + 1, nb), 256, ssmem, st>>>(
            P, n, k0, kb, cbuf[cur], cstride, piv, lu.as<double2>(), sizes, c->d_status);
        c->launches += 1;
        BGW_CUDA(c, cudaGetLastError());
      }
      {
        TimedScope tg(c, kTSweepChain, st);
        const dim3 g((n + kSolveCols - 1) / kSolveCols + (n + kCopyRows - 1) / kCopyRows, nb);
        if (sizes)
          solve_panels_kernel<true><<<g, kSolveThreads, 0, st>>>(P, n, k0, kb, lu.as<double2>(), R.as<double2>(),
                                                                 Cp.as<double2>(), sizes);
        else
          solve_panels_kernel<false><<<g, kSolveThreads, 0, st>>>(P, n, k0, kb, lu.as<double2>(), R.as<double2>(),
                                                                  Cp.as<double2>(), nullptr);
        c->launches += 1;
        BGW_CUDA(c, cudaGetLastError());
      }
      if (!oz) {
        for (int k = 0; k < nb; ++k)
          if ((rc = gj_update_run(c, P.A[k], n, k0, kb, R.as<double2>() + (size_t)k * kPB * n,
                                  Cp.as<double2>() + (size_t)k * kPB * n, st)) != BGW_OK)
            return rc;
      } else {
        TimedScope tu(c, kTOzUpdate, st);
        if ((rc = oz_slice(c, oz.get(), k0, n, 0, sizes, st)) != BGW_OK || (rc = oz_update(c, oz.get(), k0, n, 0, 0, st)) != BGW_OK)
          return rc;
        c->launches += 3;
      }
    }
    colperm_build_kernel<<<nb, 256, 2 * sizeof(int) * n, st>>>(piv, n, src);
    colperm_apply_kernel<<<dim3(n, nb), 256, sizeof(double2) * n, st>>>(P, n, src);
    BGW_CUDA(c, cudaGetLastError());
    c->launches += 2;
    m0 += nb;
  }
  return BGW_OK;
}

}  // namespace bgw
