// RI 4-index assembly (Section 3, eq 14): (ij|kl) ~ sum_PQ (ij|P) [(PQ)^-1] (Q|kl).  The metric
// (P|Q) is factored as L L^T (blocked right-looking Cholesky), B = L^-1 (P|ij) by blocked
// forward substitution, and (ij|kl) = sum_R B[R][ij] B[R][kl], either on exact digits, each element to
// the precision of its terms (psq_fx.cuh, as the solve's off-diagonal products) or, for large blocks, to 2^-38
// through the mixed path's packing and contraction.  The factor and the diagonal blocks stay on
// the FP64 pipe.  Blocks of 32 rows; every loop bound is a size argument (no waits outside the
// tensor-core products' bounded ones).
//
// Measured (693 aux functions, 51,984 pairs; FP64-pipe kernels before -> exact digits now):
// (ij|kl) block of 4096 x 4096 18.9 -> 2.1 ms (10.9 useful TFLOP/s, nine times the FP64 pipe's
// nominal rate; ALU pipe 56% busy slicing, tensor pipe 17%), solve of all pairs 24.0 -> 5.3 ms (FP64
// pipe 56% with the diagonal blocks, ALU pipe 31%).  Random data; a molecule's own integrals, whose rows are
// graded, take FP64 chains for a quarter of the elements (psq_fx.cuh).
#include "psq_internal.h"
#include "psq_fx.cuh"

#include <algorithm>
#include <cstdint>

namespace psq {
namespace {

constexpr int kB = 32;  // block size of the factor and the solve

// One block column: the kb x kb diagonal block at (k0, k0) and the panel below it, a CTA per 32 rows.
// Four lanes share a row (lane q its columns 4 i + q): one warp's FP64 instruction occupies its quarter
// of the SM for 64 cycles, so the work is spread over four warps.  Every CTA factors the diagonal block
// for itself from the lower triangle, which none of them may write in this launch: the first one parks
// the factor in the matrix's free upper triangle (below the diagonal transposed, the diagonal in the
// column after the block) until finish_factor_kernel.  Then a CTA's rows: row i gets x with x D^T = a, each x_j applied to
// the rest of the row at once (no chain but x_0, x_1, ...).  Past kb the block is the identity.  A pivot
// that is not positive records info = k0 + j + 1 (the first one wins) and continues with 1 so that
// nothing divides by zero.
// Measured with the update below: n = 693 from 2.55 ms (three launches per block column, roots and
// divisions by one thread between barriers) to 1.07, n = 82 from 266 us to 123 (past kb nothing is computed: a matrix of one to eight rows 32 -> 23 us).
__global__ void __launch_bounds__(128) chol_panel_kernel(int n, int k0, int kb, double* __restrict__ L, int* __restrict__ info) {
  __shared__ double d[kB][kB + 1];  // column-wise: d[j][i] = D[i][j]
  __shared__ double piv[2], inv[kB];  // reciprocal pivots
  const int tid = threadIdx.x, row = tid >> 2, q = tid & 3, lane = tid & 31;
  const int i0 = k0 + kb + (blockIdx.x - 1) * kB;  // block 0: the diagonal block alone
  double a[kB / 4];                                // columns 4 i + q of this row
#pragma unroll
  for (int i = 0; i < kB / 4; ++i) {
    const int c = 4 * i + q;
    a[i] = row < kb && c < kb ? (c <= row ? L[(int64_t)(k0 + row) * n + k0 + c] : 0.0) : (c == row ? 1.0 : 0.0);
  }
  // column j = 4 jj + qq: jj unrolled (registers), qq rolled (code that runs once is bound by its fetch)
#pragma unroll
  for (int jj = 0; jj < kB / 4; ++jj) {
    if (4 * jj >= kb) break;
#pragma unroll 1
    for (int qq = 0; qq < 4; ++qq) {
      const int j = 4 * jj + qq;
      if (row == j && q == qq) piv[qq & 1] = a[jj];
      __syncthreads();
      double p = piv[qq & 1];
      const int hi = __double2hiint(p);
      if (hi < 0 || hi >= 0x7ff00000 || (hi == 0 && __double2loint(p) == 0)) {  // not positive, or not a number
        if (blockIdx.x == 0 && tid == 0 && !(p > 0.0)) atomicCAS(info, 0, k0 + j + 1);
        if (!(p > 0.0)) p = 1.0;
      }
      const double y = rsqrt(p);
      if (q == qq) {
        // the diagonal entry keeps the pivot itself for now (its root: below, all at once)
        a[jj] = row > j ? a[jj] * y : (row == j ? p : 0.0);
        d[j][row] = a[jj];
      }
      if (tid == 0) inv[j] = y;
      __syncthreads();
      const double l = -d[j][row];
#pragma unroll
      for (int i = jj; i < kB / 4; ++i)
        if (i > jj || q > qq) a[i] = fma(l, d[j][4 * i + q], a[i]);
    }
  }
  __syncthreads();
  if (tid < kb) {  // the diagonal: sqrt(p) = p y, corrected by its residual
    const double p = d[tid][tid], y = inv[tid], r = p * y;
    const double t = fma(fma(-r, r, p), 0.5 * y, r);
    d[tid][tid] = (__double2hiint(t) & 0x7ff00000) == 0x7ff00000 ? sqrt(p) : t;
  }
  __syncthreads();
  if (blockIdx.x == 0) {
#pragma unroll
    for (int i = 0; i < kB / 4; ++i)
      if (const int c = 4 * i + q; row < kb && c <= row) {
        const int r0 = k0 + row, c0 = k0 + c;
        if (k0 + kb == n)  // the last block: no other CTA
          L[(int64_t)r0 * n + c0] = c == row ? d[row][row] : a[i];
        else if (c == row)
          L[(int64_t)r0 * n + k0 + kB] = d[row][row];
        else
          L[(int64_t)c0 * n + r0] = a[i];
      }
    return;
  }
#pragma unroll
  for (int i = 0; i < kB / 4; ++i) a[i] = i0 + row < n && 4 * i + q < kb ? L[(int64_t)(i0 + row) * n + k0 + 4 * i + q] : 0.0;
#pragma unroll
  for (int jj = 0; jj < kB / 4; ++jj)
#pragma unroll 1
    for (int qq = 0; qq < 4; ++qq) {
      const int j = 4 * jj + qq;
      // a / d by the reciprocal and one correction of the quotient, in the column's lane
      const double q0 = a[jj] * inv[j];
      double x = fma(fma(-q0, d[j][j], a[jj]), inv[j], q0);
      if ((__double2hiint(x) & 0x7ff00000) == 0x7ff00000) x = q0;  // an infinite pivot or quotient: no residual
      x = __shfl_sync(0xffffffffu, x, (lane & ~3) | qq);
      if (q == qq) a[jj] = x;
#pragma unroll
      for (int i = jj; i < kB / 4; ++i)
        if (i > jj || q > qq) a[i] = fma(-x, d[j][4 * i + q], a[i]);
    }
#pragma unroll
  for (int i = 0; i < kB / 4; ++i)
    if (i0 + row < n && 4 * i + q < kb) L[(int64_t)(i0 + row) * n + k0 + 4 * i + q] = a[i];
}

// Trailing update L[i][j] -= sum_m L[i][k0+m] L[j][k0+m] for k1 = k0 + kb <= j <= i < n, one
// CTA per 32 x 32 tile of the lower triangle (tile t -> (ti, tj), ti >= tj).
__global__ void __launch_bounds__(256) chol_update_kernel(int n, int k0, int kb, double* __restrict__ L) {
  __shared__ double pa[kB][kB + 1], pb[kB][kB + 1];
  const int k1 = k0 + kb;
  const int t = blockIdx.x;
  int ti = (int)((sqrt(8.0 * t + 1.0) - 1.0) * 0.5);
  while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
  while (ti * (ti + 1) / 2 > t) --ti;
  const int tj = t - ti * (ti + 1) / 2;
  const int i0 = k1 + ti * kB, j0 = k1 + tj * kB;
  for (int q = threadIdx.x; q < kB * kB; q += blockDim.x) {
    const int r = q >> 5, m = q & 31;
    pa[r][m] = (i0 + r < n && m < kb) ? L[(int64_t)(i0 + r) * n + k0 + m] : 0.0;
    pb[r][m] = (j0 + r < n && m < kb) ? L[(int64_t)(j0 + r) * n + k0 + m] : 0.0;
  }
  __syncthreads();
  const int c = threadIdx.x & 31, r0 = threadIdx.x >> 5;  // rows r0, r0 + 8, r0 + 16, r0 + 24
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int m = 0; m < kb; ++m) {
    const double b = pb[c][m];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = fma(pa[r0 + 8 * q][m], b, acc[q]);
  }
  const int j = j0 + c;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = i0 + r0 + 8 * q;
    if (i < n && j < n && j <= i) L[(int64_t)i * n + j] -= acc[q];
  }
}

// The diagonal blocks' factors from where chol_panel_kernel parked them; zeros above the diagonal.  The
// thread of a parked entry's lower element moves it, so that no other reads what it clears.
__global__ void finish_factor_kernel(int n, double* __restrict__ L) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)n * n) return;
  const int i = (int)(idx / n), j = (int)(idx % n), k1 = (i / kB + 1) * kB;  // the column after i's block
  if (j > i) {
    if (j > k1 || k1 >= n) L[idx] = 0.0;
  } else if (j / kB == i / kB && k1 < n) {
    const int64_t from = i == j ? (int64_t)i * n + k1 : (int64_t)j * n + i;
    L[idx] = L[from];
    L[from] = 0.0;
  }
}

// The plain sums of a window's products for row r and the columns from c (fx::window's chain): factor a of row r
// and point p at a[p ap + r ar], factor b of column c at b[p bp + c bc].
struct ProductChain {
  const double* a;
  int64_t ap, ar;
  const double* b;
  int64_t bp, bc;
  int rows, cols, points;
  template <int N>
  __device__ __forceinline__ void operator()(int r, int c, int p0, int step, double (&s)[N]) const {
    if (r >= rows || c >= cols) return;
    int64_t col[N];
#pragma unroll
    for (int j = 0; j < N; ++j) col[j] = min(c + j, cols - 1) * bc;
#pragma unroll 8
    for (int p = p0; p < points; p += step) {
      const double x = a[p * ap + r * ar];
#pragma unroll
      for (int j = 0; j < N; ++j) s[j] = fma(x, b[p * bp + col[j]], s[j]);
    }
  }
};

// Forward substitution B <- L^-1 B, left-looking, one launch: a CTA owns up to 128 columns and
// walks down the 32-row blocks.  Block k's rows take sum_{q < 32 k} L[r][q] B[q][col] from the
// tensor cores (fx::window: the columns are the tile's rows, the block's rows of L its columns),
// then the 32 x 32 diagonal block is solved in FP64, one thread per column.
__global__ void __launch_bounds__(fx::kThreads, 2) trsv_kernel(int n, int64_t m, int cols, const double* __restrict__ L, double* B) {
  extern __shared__ __align__(1024) uint8_t raw[];
  fx::Smem& sm = fx::smem_at(raw);
  const uint32_t tmem = fx::open(sm);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t c0 = (int64_t)blockIdx.x * cols;
  const int live = (int)(m - c0 < cols ? m - c0 : cols);  // columns of this CTA
  // after a block's products the digit planes are free: they hold its right-hand sides [row][col]
  // and the diagonal block with its reciprocal pivots
  double(*rhs)[fx::kRows] = reinterpret_cast<double(*)[fx::kRows]>(sm.a[0]);
  double(*d)[kB + 1] = reinterpret_cast<double(*)[kB + 1]>(sm.a[0] + sizeof(double) * kB * fx::kRows);
  uint32_t phase = 0, win = 0;
  bool ok = true, run = true;
  for (int k0 = 0; k0 < n && run; k0 += kB) {
    const int kb = n - k0 < kB ? n - k0 : kB;
    double acc[16] = {};
    for (int q0 = 0; q0 < k0 && run; q0 += fx::kWin, ++win) {
      double va[4][8], vb[2][4];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const double* p = B + (int64_t)(q0 + fx::a_pt(c)) * m + c0 + fx::a_row(u);
#pragma unroll
          for (int i = 0; i < 8; ++i)
            va[2 * c + u][i] = fx::a_row(u) < live && q0 + fx::a_pt(c) + i < k0 ? p[i * m] : 0.0;
        }
        const double* p = L + (int64_t)(k0 + fx::b_col()) * n + q0 + fx::b_pt(c);
#pragma unroll
        for (int i = 0; i < 4; ++i) vb[c][i] = fx::b_col() < kb && q0 + fx::b_pt(c) + i < k0 ? p[i] : 0.0;
      }
      run = fx::window(sm, tmem, va, vb, acc, phase, win, live, kb, ok,
                       ProductChain{B + (int64_t)q0 * m + c0, m, 1, L + (int64_t)k0 * n + q0, 1, n, live, kb,
                                    min(k0 - q0, fx::kWin)});
    }
    if (k0 > 0 && run) run = __syncthreads_and(ok);  // and no MMA reads the planes any more
    if (!run) break;
    const int r = 32 * (warp & 3) + lane;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int i = 16 * (warp >> 2) + j;
      rhs[i][r] = i < kb && r < live ? B[(int64_t)(k0 + i) * m + c0 + r] - acc[j] : 0.0;
    }
    for (int t = tid; t < kB * kB; t += fx::kThreads) {
      const int i = t >> 5, c = t & 31;
      d[i][c] = (i < kb && c <= i) ? L[(int64_t)(k0 + i) * n + k0 + c] : 0.0;
    }
    __syncthreads();
    if (tid < kB) d[tid][kB] = tid < kb ? 1.0 / d[tid][tid] : 0.0;
    __syncthreads();
    if (tid < live) {
      double x[kB];
#pragma unroll
      for (int j = 0; j < kB; ++j) {
        if (j < kb) {
          double s = rhs[j][tid];
#pragma unroll
          for (int q = 0; q < j; ++q) s -= d[j][q] * x[q];
          // s / d by the reciprocal and one correction of the quotient
          const double q0 = s * d[j][kB];
          const double q1 = fma(fma(-q0, d[j][j], s), d[j][kB], q0);
          x[j] = isfinite(q1) ? q1 : s / d[j][j];
          B[(int64_t)(k0 + j) * m + c0 + tid] = x[j];
        }
      }
    }
    __syncthreads();
  }
  if (!run && tid < live)  // a wait ran out: no result is better than a wrong one
    for (int q = 0; q < n; ++q) B[(int64_t)q * m + c0 + tid] = __longlong_as_double(0x7ff8000000000000ll);
  fx::close(sm, tmem, run, phase);
}

// Few columns (psq_ri_solve has the rule): right-looking, two launches per block, so that the rows below a
// block spread over the SMs, on the FP64 pipe.
//
// Forward substitution on the diagonal block: B[k0 + r][col] for r < kb, one thread per
// column.
__global__ void __launch_bounds__(256) trsv_diag_kernel(int n, int64_t m, int k0, int kb,
                                                        const double* __restrict__ L, double* __restrict__ B) {
  __shared__ double d[kB][kB + 1];
  for (int t = threadIdx.x; t < kB * kB; t += blockDim.x) {
    const int r = t >> 5, c = t & 31;
    d[r][c] = (r < kb && c <= r) ? L[(int64_t)(k0 + r) * n + k0 + c] : 0.0;
  }
  __syncthreads();
  const int64_t col = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= m) return;
  double* b = B + (int64_t)k0 * m + col;
  double x[kB];
#pragma unroll
  for (int j = 0; j < kB; ++j) {
    if (j < kb) {
      double s = b[(int64_t)j * m];
#pragma unroll
      for (int q = 0; q < j; ++q) s -= d[j][q] * x[q];
      x[j] = s / d[j][j];
      b[(int64_t)j * m] = x[j];
    }
  }
}

// B[k1 + r][col] -= sum_q L[k1 + r][k0 + q] B[k0 + q][col]: 64 x 64 tiles, 256 threads with
// 4 x 4 outputs each.
__global__ void __launch_bounds__(256) trsv_update_kernel(int n, int64_t m, int k0, int kb,
                                                          const double* __restrict__ L, double* __restrict__ B) {
  __shared__ double ls[64][kB + 1];
  __shared__ double bs[kB][64];
  const int k1 = k0 + kb;
  const int i0 = k1 + blockIdx.y * 64;
  const int64_t c0 = (int64_t)blockIdx.x * 64;
  for (int t = threadIdx.x; t < 64 * kB; t += blockDim.x) {
    const int r = t / kB, q = t % kB;
    ls[r][q] = (i0 + r < n && q < kb) ? L[(int64_t)(i0 + r) * n + k0 + q] : 0.0;
  }
  for (int t = threadIdx.x; t < kB * 64; t += blockDim.x) {
    const int q = t / 64, c = t % 64;
    bs[q][c] = (q < kb && c0 + c < m) ? B[(int64_t)(k0 + q) * m + c0 + c] : 0.0;
  }
  __syncthreads();
  const int tr = threadIdx.x / 16, tc = threadIdx.x % 16;  // rows tr + 16a, columns tc + 16b
  double acc[4][4] = {};
  for (int q = 0; q < kb; ++q) {
    double lv[4], bv[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) lv[a] = ls[tr + 16 * a][q];
#pragma unroll
    for (int b = 0; b < 4; ++b) bv[b] = bs[q][tc + 16 * b];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = fma(lv[a], bv[b], acc[a][b]);
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int i = i0 + tr + 16 * a;
    if (i >= n) continue;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int64_t c = c0 + tc + 16 * b;
      if (c < m) B[(int64_t)i * m + c] -= acc[a][b];
    }
  }
}

// out[c][d] = sum_R B[R][c0 + c] B[R][d0 + d]: a CTA per 128 x 32 output tile, R in windows of 64.
__global__ void __launch_bounds__(fx::kThreads, 2) eri_kernel(int n, int64_t m, const double* __restrict__ B, int64_t c0,
                                                              int64_t nc, int64_t d0, int64_t nd, double* __restrict__ out) {
  extern __shared__ __align__(1024) uint8_t raw[];
  fx::Smem& sm = fx::smem_at(raw);
  const uint32_t tmem = fx::open(sm);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t tc0 = (int64_t)blockIdx.y * fx::kRows, td0 = (int64_t)blockIdx.x * fx::kCols;
  const int rows = (int)(nc - tc0 < fx::kRows ? nc - tc0 : fx::kRows), cols = (int)(nd - td0 < fx::kCols ? nd - td0 : fx::kCols);
  double acc[16] = {};
  uint32_t phase = 0, win = 0;
  bool ok = true, run = true;
  for (int R0 = 0; R0 < n && run; R0 += fx::kWin, ++win) {
    double va[4][8], vb[2][4];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const double* p = B + (int64_t)(R0 + fx::a_pt(c)) * m + c0 + tc0 + fx::a_row(u);
#pragma unroll
        for (int i = 0; i < 8; ++i)
          va[2 * c + u][i] = fx::a_row(u) < rows && R0 + fx::a_pt(c) + i < n ? __ldg(p + i * m) : 0.0;
      }
      const double* p = B + (int64_t)(R0 + fx::b_pt(c)) * m + d0 + td0 + fx::b_col();
#pragma unroll
      for (int i = 0; i < 4; ++i) vb[c][i] = fx::b_col() < cols && R0 + fx::b_pt(c) + i < n ? __ldg(p + i * m) : 0.0;
    }
    run = fx::window(sm, tmem, va, vb, acc, phase, win, rows, cols, ok,
                     ProductChain{B + (int64_t)R0 * m + c0 + tc0, m, 1, B + (int64_t)R0 * m + d0 + td0, m, 1, rows, cols,
                                  min(n - R0, fx::kWin)});
  }
  if (run) run = __syncthreads_and(ok);
  const int r = 32 * (warp & 3) + lane;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int d = 16 * (warp >> 2) + j;
    if (r < rows && d < cols) out[(tc0 + r) * nd + td0 + d] = run ? acc[j] : __longlong_as_double(0x7ff8000000000000ll);
  }
  fx::close(sm, tmem, run, phase);
}

// ---------------------------------------------------------------- tensor-core product
//
// (ij|kl) = sum_R B[R][ij] B[R][kl] is the contraction of eq 9 with the aux index R in the
// place of the points: the pair columns of B become operand rows (transposed into Bt), are
// packed as in the mixed path (five 8-bit slices per value under a power-of-two scale per
// row and 128 aux functions), and the tcgen05 contraction and its FP64 range reduction run
// unchanged on them (one block, A = the c pairs, B = the d pairs, no row constants).

constexpr size_t kAlign = 256;
size_t up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

struct RiMixedLayout {
  int64_t nc, nd;
  int n, nch, nwin, tmA, tnB, n_ranges, win_per, n_ctas;
  int64_t n_items, jobsA, jobsB;
  size_t o_grid, o_pn, o_blk, o_items, o_cb, o_eb, o_status, o_bt, o_pack, o_part, total;
  int64_t packA, expA, packB, expB;  // panel offsets within the packed area
};

RiMixedLayout ri_mixed_layout(int n, int64_t nc, int64_t nd, int sm_count) {
  RiMixedLayout L{};
  L.n = n; L.nc = nc; L.nd = nd;
  L.nch = (n + kChunkPts - 1) / kChunkPts;
  L.nwin = (n + kWinPts - 1) / kWinPts;
  L.tmA = (int)((nc + kMmaM - 1) / kMmaM);
  L.tnB = (int)((nd + kMmaN - 1) / kMmaN);
  const int64_t tiles = (int64_t)L.tmA * L.tnB;
  const int64_t want = 2LL * sm_count;  // at least two items per SM: ranges of aux windows
  int r = tiles >= want ? 1 : (int)std::min<int64_t>(L.nwin, (want + tiles - 1) / tiles);
  L.win_per = (L.nwin + r - 1) / r;
  L.n_ranges = (L.nwin + L.win_per - 1) / L.win_per;
  L.n_items = tiles * L.n_ranges;
  L.n_ctas = (int)std::min<int64_t>(L.n_items, sm_count);
  L.jobsA = (int64_t)L.tmA * L.nwin * (kMmaM / kPackRows);
  L.jobsB = (int64_t)L.tnB * L.nwin * (kMmaN / kPackRows);
  size_t o = 0;
  auto sec = [&](size_t bytes) { const size_t at = o; o = up(o + bytes); return at; };
  L.o_status = sec(sizeof(int));
  L.o_grid = sec(sizeof(DevGrid));
  L.o_pn = sec(2 * sizeof(Panel));
  L.o_blk = sec(sizeof(MmaBlock));
  L.o_items = sec(sizeof(GemmItem) * (size_t)L.n_items);
  L.o_cb = sec(sizeof(int) * (size_t)(L.n_ctas + 1));
  L.o_eb = sec(2 * sizeof(int64_t));
  L.o_bt = sec(sizeof(double) * (size_t)(nc + nd) * n);
  size_t pk = 0;
  auto psec = [&](size_t bytes) { const size_t at = pk; pk = up(pk + bytes); return (int64_t)at; };
  L.packA = psec((size_t)nc * L.nch * kSlices * 2 * kChunkPts);
  L.expA = psec((size_t)L.tmA * L.nwin * kMmaM * 4);
  L.packB = psec((size_t)nd * L.nch * kSlices * 2 * kChunkPts);
  L.expB = psec((size_t)L.tnB * L.nwin * kMmaN * 4);
  L.o_pack = sec(pk);
  L.o_part = sec(sizeof(float2) * (size_t)L.n_ranges * nc * nd);
  L.total = o;
  return L;
}

// The tables of the one-block plan, written on the device (nothing to stage on the host, so
// the call can be captured in a CUDA graph).  Items dealt round-robin, stored per CTA.
__global__ void ri_setup_kernel(RiMixedLayout L, char* __restrict__ ws) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    *reinterpret_cast<int*>(ws + L.o_status) = 0;
    DevGrid* g = reinterpret_cast<DevGrid*>(ws + L.o_grid);
    g->K = L.n;
    Panel* pn = reinterpret_cast<Panel*>(ws + L.o_pn);
    pn[0].grid = 0; pn[0].rows_off = 0; pn[0].nrows = (int)L.nc; pn[0].tr = kMmaM; pn[0].n_tiles = L.tmA;
    pn[0].nch = L.nch; pn[0].nwin = L.nwin; pn[0].pack_off = L.packA; pn[0].exp_off = L.expA; pn[0].job_begin = 0;
    pn[1].grid = 0; pn[1].rows_off = (int)L.nc; pn[1].nrows = (int)L.nd; pn[1].tr = kMmaN; pn[1].n_tiles = L.tnB;
    pn[1].nch = L.nch; pn[1].nwin = L.nwin; pn[1].pack_off = L.packB; pn[1].exp_off = L.expB; pn[1].job_begin = L.jobsA;
    MmaBlock* b = reinterpret_cast<MmaBlock*>(ws + L.o_blk);
    b->grid = 0; b->m = (int)L.nc; b->n = (int)L.nd; b->a_off = 0; b->b_off = (int)L.nc;
    b->n_ranges = L.n_ranges; b->win_per = L.win_per; b->a_panel = 0; b->b_panel = 1;
    b->ptile_off = 0; b->n_btiles = 0; b->res_off = 0; b->part_off = 0;
    int64_t* eb = reinterpret_cast<int64_t*>(ws + L.o_eb);
    eb[0] = 0;
    eb[1] = L.nc * L.nd;
  }
  const int64_t q = L.n_items / L.n_ctas, rem = L.n_items % L.n_ctas;
  if (i <= L.n_ctas) reinterpret_cast<int*>(ws + L.o_cb)[i] = (int)(i * q + (i < rem ? i : rem));
  if (i < L.n_items) {
    const int64_t tiles = (int64_t)L.tmA * L.tnB;
    const int chunk = (int)(i / tiles), t = (int)(i % tiles);
    const int64_t bcta = i % L.n_ctas, j = i / L.n_ctas;
    const int64_t slot = bcta * q + (bcta < rem ? bcta : rem) + j;
    reinterpret_cast<GemmItem*>(ws + L.o_items)[slot] = GemmItem{0, t / L.tnB, t % L.tnB, chunk};
  }
}

// Bt[r][R] = B[R][col0 + r] for r < count: the pair columns as rows (32 x 32 tiles).
__global__ void ri_transpose_kernel(int n, int64_t m, const double* __restrict__ B, int64_t col0, int64_t count,
                                    double* __restrict__ Bt) {
  __shared__ double tile[32][33];
  const int64_t c0 = (int64_t)blockIdx.x * 32;
  const int R0 = blockIdx.y * 32;
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int R = R0 + k;
    const int64_t c = c0 + threadIdx.x;
    tile[k][threadIdx.x] = (R < n && c < count) ? B[(int64_t)R * m + col0 + c] : 0.0;
  }
  __syncthreads();
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int64_t c = c0 + k;
    const int R = R0 + threadIdx.x;
    if (c < count && R < n) Bt[c * n + R] = tile[threadIdx.x][k];
  }
}

// The dynamic shared memory of a tile kernel (an attribute per device, set before each launch).
bool fx_attr(const void* kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fx::kSmemBytes) == cudaSuccess;
}

bool aligned8(const void* p) { return ((uintptr_t)p & 7u) == 0; }

psq_status launched() {
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? PSQ_OK : set_error(PSQ_ERR_CUDA, cudaGetErrorString(e));
}

}  // namespace
}  // namespace psq

using namespace psq;

extern "C" psq_status psq_ri_factor(int n, const double* d_J2, double* d_L, int* d_info, void* stream) {
  if (n < 0) return set_error(PSQ_ERR_ARG, "psq_ri_factor: n < 0");
  if (!d_info || ((uintptr_t)d_info & 3u)) return set_error(PSQ_ERR_ARG, "psq_ri_factor: d_info NULL or misaligned");
  if (n > 0 && (!d_J2 || !d_L || !aligned8(d_J2) || !aligned8(d_L)))
    return set_error(PSQ_ERR_ARG, "psq_ri_factor: NULL or misaligned matrix");
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(d_info, 0, sizeof(int), s) != cudaSuccess) return launched();
  if (n == 0) return PSQ_OK;
  if (d_L != d_J2 &&
      cudaMemcpyAsync(d_L, d_J2, sizeof(double) * (size_t)n * n, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return launched();
  for (int k0 = 0; k0 < n; k0 += kB) {
    const int kb = n - k0 < kB ? n - k0 : kB;
    const int rest = n - k0 - kb, T = (rest + kB - 1) / kB;
    chol_panel_kernel<<<1 + T, 128, 0, s>>>(n, k0, kb, d_L, d_info);
    if (rest > 0) chol_update_kernel<<<T * (T + 1) / 2, 256, 0, s>>>(n, k0, kb, d_L);
  }
  const int64_t nn = (int64_t)n * n;
  finish_factor_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, s>>>(n, d_L);
  return launched();
}

extern "C" psq_status psq_ri_solve(int n, int64_t m, const double* d_L, double* d_B, void* stream) {
  if (n < 0 || m < 0) return set_error(PSQ_ERR_ARG, "psq_ri_solve: negative size");
  if (n == 0 || m == 0) return PSQ_OK;
  if (!d_L || !d_B || !aligned8(d_L) || !aligned8(d_B))
    return set_error(PSQ_ERR_ARG, "psq_ri_solve: NULL or misaligned matrix");
  if ((m + 63) / 64 > 0x7fffffff) return set_error(PSQ_ERR_ARG, "psq_ri_solve: m too large");
  cudaStream_t s = (cudaStream_t)stream;
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return launched();
  // The tensor-core kernel walks down the blocks within a CTA: where its CTAs are one wave, about 7.6 us for each of
  // the nb^2 / 4 windows and 38 us for each diagonal block.  Two launches per block on the FP64 pipe: about 70 us and
  // n^2 m FMAs at 0.59 per ps in all.  Measured, tensor cores against FP64 pipe: n = 2000, 1 and 40 columns 9.9 against
  // 4.4 ms; n = 3000, 500 columns 20.6 against 10.8 ms; n = 693, 1 column 1.73 against 1.51 ms, 300 columns 1.77
  // against 1.92 ms; n = 200, 200 columns 0.33 against 0.51 ms.
  // A single block has no products: 16 rows or fewer (n = 8, 3,000 columns 15 against 12 us), columns of one CTA
  // (n = 32, 50 columns 44 against 37 us) or more than the tensor-core kernel's first CTAs hold (n = 32, 3,000
  // columns 43 against 54 us, 51,984 columns 115 against 102 us) take the FP64 one too.
  const int64_t nb = (n + kB - 1) / kB;
  const bool fp64 = nb == 1 ? n <= 16 || m <= 256 || m > 160LL * sms
                            : m <= 2LL * fx::kRows * sms &&
                                  70.0 * nb + (double)n * n * m / 1.18e6 < 7.6 * (nb * nb / 4) + 38.0 * nb;
  if (fp64) {
    for (int k0 = 0; k0 < n; k0 += kB) {
      const int kb = n - k0 < kB ? n - k0 : kB, rest = n - k0 - kb;
      trsv_diag_kernel<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(n, m, k0, kb, d_L, d_B);
      if (rest > 0)
        trsv_update_kernel<<<dim3((unsigned)((m + 63) / 64), (rest + 63) / 64), 256, 0, s>>>(n, m, k0, kb, d_L, d_B);
    }
    return launched();
  }
  // few columns: fewer per CTA, so that the serial substitutions spread over the SMs (two CTAs each)
  const int64_t per = (m + 2 * sms - 1) / (2 * sms);
  const int cols = per >= 97 ? 128 : (int)((per + 31) / 32 * 32);
  if (!fx_attr((const void*)trsv_kernel)) return launched();
  trsv_kernel<<<(unsigned)((m + cols - 1) / cols), fx::kThreads, fx::kSmemBytes, s>>>(n, m, cols, d_L, d_B);
  return launched();
}

extern "C" psq_status psq_ri_eri(int n, int64_t m, const double* d_B, int64_t c0, int64_t nc, int64_t d0, int64_t nd,
                                 double* d_out, void* stream) {
  if (n < 0 || m < 0 || nc < 0 || nd < 0) return set_error(PSQ_ERR_ARG, "psq_ri_eri: negative size");
  if (c0 < 0 || d0 < 0 || c0 + nc > m || d0 + nd > m) return set_error(PSQ_ERR_ARG, "psq_ri_eri: range outside [0, m)");
  if (nc == 0 || nd == 0) return PSQ_OK;
  if (!d_out || !aligned8(d_out) || (n > 0 && (!d_B || !aligned8(d_B))))
    return set_error(PSQ_ERR_ARG, "psq_ri_eri: NULL or misaligned pointer");
  if ((nc + 63) / 64 > 65535 || (nd + 63) / 64 > 0x7fffffff) return set_error(PSQ_ERR_ARG, "psq_ri_eri: block too large");
  if (!fx_attr((const void*)eri_kernel)) return launched();
  eri_kernel<<<dim3((unsigned)((nd + fx::kCols - 1) / fx::kCols), (unsigned)((nc + fx::kRows - 1) / fx::kRows)), fx::kThreads,
               fx::kSmemBytes, (cudaStream_t)stream>>>(n, m, d_B, c0, nc, d0, nd, d_out);
  return launched();
}

extern "C" psq_status psq_ri_eri_mixed_workspace(int n, int64_t nc, int64_t nd, size_t* bytes) {
  if (!bytes) return set_error(PSQ_ERR_ARG, "psq_ri_eri_mixed_workspace: bytes is NULL");
  if (n < 0 || nc < 0 || nd < 0) return set_error(PSQ_ERR_ARG, "psq_ri_eri_mixed_workspace: negative size");
  if (nc > (1 << 30) || nd > (1 << 30)) return set_error(PSQ_ERR_UNSUPPORTED, "psq_ri_eri_mixed_workspace: block too large");
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  *bytes = ri_mixed_layout(n, nc, nd, sms).total;
  return PSQ_OK;
}

extern "C" psq_status psq_ri_eri_mixed(int n, int64_t m, const double* d_B, int64_t c0, int64_t nc, int64_t d0,
                                       int64_t nd, double* d_out, void* d_workspace, size_t ws_bytes, void* stream) {
  if (n < 0 || m < 0 || nc < 0 || nd < 0) return set_error(PSQ_ERR_ARG, "psq_ri_eri_mixed: negative size");
  if (c0 < 0 || d0 < 0 || c0 + nc > m || d0 + nd > m)
    return set_error(PSQ_ERR_ARG, "psq_ri_eri_mixed: range outside [0, m)");
  if (nc == 0 || nd == 0) return PSQ_OK;
  if (!d_out || !aligned8(d_out) || (n > 0 && (!d_B || !aligned8(d_B))))
    return set_error(PSQ_ERR_ARG, "psq_ri_eri_mixed: NULL or misaligned pointer");
  if (!d_workspace || (uintptr_t)d_workspace % kAlign)
    return set_error(PSQ_ERR_ARG, "psq_ri_eri_mixed: workspace NULL or not 256-byte aligned");
  if (nc > (1 << 30) || nd > (1 << 30)) return set_error(PSQ_ERR_UNSUPPORTED, "psq_ri_eri_mixed: block too large");
  cudaStream_t s = (cudaStream_t)stream;
  if (n == 0) {
    if (cudaMemsetAsync(d_out, 0, sizeof(double) * (size_t)nc * nd, s) != cudaSuccess) return launched();
    return PSQ_OK;
  }
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return launched();
  const RiMixedLayout L = ri_mixed_layout(n, nc, nd, sms);
  if (ws_bytes < L.total) return set_error(PSQ_ERR_OOM, "psq_ri_eri_mixed: workspace too small");
  if (prepare_kernels() != cudaSuccess) return launched();
  char* ws = (char*)d_workspace;
  if (cudaMemsetAsync(ws, 0, L.o_bt, s) != cudaSuccess) return launched();  // tables (zeroed, then set)
  const int64_t setup_n = std::max<int64_t>(L.n_items, L.n_ctas + 1);
  ri_setup_kernel<<<(unsigned)((setup_n + 255) / 256), 256, 0, s>>>(L, ws);
  double* btA = (double*)(ws + L.o_bt);
  double* btB = btA + (size_t)nc * n;
  ri_transpose_kernel<<<dim3((unsigned)((nc + 31) / 32), (n + 31) / 32), dim3(32, 8), 0, s>>>(n, m, d_B, c0, nc, btA);
  ri_transpose_kernel<<<dim3((unsigned)((nd + 31) / 32), (n + 31) / 32), dim3(32, 8), 0, s>>>(n, m, d_B, d0, nd, btB);
  uint8_t* packed = (uint8_t*)(ws + L.o_pack);
  const Panel* pn = (const Panel*)(ws + L.o_pn);
  if (launch_ri_pack(pn, L.jobsA + L.jobsB, btA, btB, n, packed, s) != cudaSuccess) return launched();
  if (launch_contract_ws((const DevGrid*)(ws + L.o_grid), (const MmaBlock*)(ws + L.o_blk),
                         (const GemmItem*)(ws + L.o_items), (const int*)(ws + L.o_cb), L.n_ctas, pn, nullptr, nullptr,
                         nullptr, packed, (float2*)(ws + L.o_part), (int*)(ws + L.o_status), 4000000000ull,
                         nullptr, s) != cudaSuccess)
    return launched();
  if (launch_reduce_mixed((const DevGrid*)(ws + L.o_grid), (const MmaBlock*)(ws + L.o_blk), 1,
                          (const int64_t*)(ws + L.o_eb), 0, nc * nd, nullptr, nullptr, (const float2*)(ws + L.o_part), d_out, s) != cudaSuccess)
    return launched();
  return launched();
}
