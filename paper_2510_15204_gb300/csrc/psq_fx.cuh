// FP64 sums of products on the tensor cores, without rounding the products: per window of 64
// points, R[r][c] += sum_p a_r(p) b_c(p) for a tile of 128 rows x 32 columns, by a CTA of 256
// threads.
//
// GB300's FP64 pipe does two FMAs per clock and SM (1.25 TFLOP/s), its tensor cores 4096 16-bit
// ones.  So every value is cut, without rounding error, into integer digits (the error-free split
// of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59 (2012), here with one power-of-two scale
// per row and window).  With |v| < 2^e over the window, X = trunc(v 2^(62-e)) is a 63-bit integer,
// written as eight balanced base-256 digits d_k in [-128, 127] (|d_0| <= 64), exact in FP16.
// The products of orders i + j = 0..7 (36 of 64) accumulate per order in FP32: an order's sum over
// 64 points stays below 64 x 8 x 2^14 = 2^23, so the accumulation is exact.  The order sums join
// in one 64-bit integer T with unit 2^(ea+eb-52), and the FP64 accumulator of an element takes
// T by one FMA per window: where a chain of FP64 FMAs rounds 64 times, this rounds once.  What is
// dropped (the truncation of X, orders above 7, the fraction of orders 6 and 7 below T's unit)
// stays below two units per window, 2^-51 of the largest |a| times the largest |b|, against 2^-53
// of the running sum per FMA of the chain.
//
// Rows whose window lies below 2^-958 count as zeros.  Rows that hold an infinity, a NaN or a value of 2^478 and above take the plain FP64 chain for the
// window (their products with the other operand may leave the range of the integer path).
//
// Layout.  Two CTAs per SM (82 KB of shared memory and 256 of the 512 TMEM columns each), so that
// one slices or folds while the other's MMAs run.  The digits of 32 points are eight planes of
// 64-byte rows in the 64-byte swizzle (A: 8 x 8 KB, B: 8 x 2 KB); the B planes are contiguous, so
// A plane i against B planes 0..7-i is one MMA of N = 32 (8 - i) whose columns land on the order
// accumulators i..7.
#pragma once
#include <cuda_fp16.h>

#include "psq_tc.cuh"

namespace psq {
namespace fx {

constexpr int kThreads = 256;
constexpr int kRows = 128, kCols = 32;  // tile of a CTA
constexpr int kWin = 64;                // points per scale window
constexpr int kDigits = 8;
constexpr uint32_t kTmemCols = kDigits * kCols;
constexpr int kBigField = 1500;         // exponent field from which a row takes the FP64 chain

struct Smem {
  alignas(1024) uint8_t a[kDigits][kRows * 64];
  alignas(1024) uint8_t b[kDigits][kCols * 64];
  int ma[2][kRows];  // largest |high word| of the two threads of a row
  int mb[8][kCols];  // and of the eight threads of a column
  int ea[kRows], eb[kCols];  // exponent fields of the window
  alignas(8) uint64_t done;
  uint32_t tmem;
};
constexpr size_t kSmemBytes = sizeof(Smem) + 1024;

// Instruction descriptor: kind::f16, A = B = F16, D = F32, both K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t idesc(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);
}

__device__ __forceinline__ Smem& smem_at(uint8_t* raw) {
  return *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~(uintptr_t)1023);
}

// Start and end of a CTA's use (all threads).
__device__ __forceinline__ uint32_t open(Smem& sm) {
  if (threadIdx.x < 32) mma::tmem_alloc(&sm.tmem, kTmemCols);
  if (threadIdx.x == 0) {
    mma::mbar_init(&sm.done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  mma::fence_before();
  __syncthreads();
  mma::fence_after();
  return sm.tmem;
}
__device__ __forceinline__ void close(Smem& sm, uint32_t tmem, bool ok, uint32_t phase) {
  if (!ok) mma::mbar_wait(mma::smem_u32(&sm.done), phase & 1);  // the MMAs still in flight
  mma::fence_before();
  __syncthreads();
  if (threadIdx.x < 32) {
    mma::fence_after();
    mma::tmem_free(tmem, kTmemCols);
  }
}

// The operand values a thread brings to a window: row threadIdx.x % 128, points
// 32 c + 16 (threadIdx.x / 128) + i of chunk c (a[16 c + i]); column threadIdx.x % 32, points
// 8 (threadIdx.x / 32) + i (b[i]).
__device__ __forceinline__ int a_row() { return threadIdx.x & (kRows - 1); }
__device__ __forceinline__ int a_pt(int c) { return 32 * c + 16 * (threadIdx.x >> 7); }
__device__ __forceinline__ int b_col() { return threadIdx.x & (kCols - 1); }
__device__ __forceinline__ int b_pt() { return 8 * (threadIdx.x >> 5); }

// Biased digits of v (byte k of the result = digit 7 - k plus 128) in a window whose largest
// exponent field is E (E = 4000: a row of zeros).
__device__ __forceinline__ uint64_t digits(double v, int E) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const int t = min(E - (int)((hi >> 20) & 0x7ffu), 63);
  const uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  const uint64_t x = (m << 9) >> t;
  const uint64_t s = (uint64_t)((int64_t)(int32_t)hi >> 63);
  return ((x ^ s) - s) + 0x8080808080808080ull;
}

// Eight consecutive points of one row or column into its 16-byte group of every plane.
__device__ __forceinline__ void store_group(uint8_t* planes, uint32_t plane_bytes, uint32_t off, const double* v, int E) {
  uint64_t y[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) y[i] = digits(v[i], E);
  const __half2 bias = __half2half2(__ushort_as_half(0x6480));  // 1024 + 128
#pragma unroll
  for (int k = 0; k < kDigits; ++k) {
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t u0 = k < 4 ? (uint32_t)(y[2 * q] >> 32) : (uint32_t)y[2 * q];
      const uint32_t u1 = k < 4 ? (uint32_t)(y[2 * q + 1] >> 32) : (uint32_t)y[2 * q + 1];
      const uint32_t by = 3 - (k & 3);
      // 1024 + byte in both halves, then minus 1152: the digit, exact in FP16
      const uint32_t x = (__byte_perm(u0, u1, by | (by << 4) | ((4 + by) << 8) | ((4 + by) << 12)) & 0x00ff00ffu) | 0x64006400u;
      const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&x), bias);
      w[q] = *reinterpret_cast<const uint32_t*>(&d);
    }
    *reinterpret_cast<uint4*>(planes + k * plane_bytes + off) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

__device__ __forceinline__ int hi_abs(double v) { return __double2hiint(v) & 0x7fffffff; }

// One window: the tile's accumulators (element row 32 (warp % 4) + lane, columns 16 (warp / 4) + j,
// acc[j]) take sum_p a_r(p) b_c(p).  phase: the parity of sm.done, kept by the caller from 0.
// chain(row, col): the plain FP64 sum of the window for a row or column out of the integer
// path's range.  Returns false (for every thread) when a wait ran out.
template <typename Chain>
__device__ __forceinline__ bool window(Smem& sm, uint32_t tmem, const double (&va)[32], const double (&vb)[8],
                                       double (&acc)[16], uint32_t& phase, Chain chain) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int ma = 0, mb = 0;
#pragma unroll
  for (int i = 0; i < 32; ++i) ma = max(ma, hi_abs(va[i]));
#pragma unroll
  for (int i = 0; i < 8; ++i) mb = max(mb, hi_abs(vb[i]));
  sm.ma[tid >> 7][tid & 127] = ma;
  sm.mb[warp][lane] = mb;
  __syncthreads();
  const int Ea = max(sm.ma[0][tid & 127], sm.ma[1][tid & 127]) >> 20;
  int Eb = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) Eb = max(Eb, sm.mb[i][lane]);
  Eb >>= 20;
  if (tid < kRows) sm.ea[tid] = Ea;
  if (tid < kCols) sm.eb[tid] = Eb;
  // rows below 2^-958 count as zeros (a zero's own field, 0, is then at least 64 below E)
  const int Sa = Ea >= 64 ? Ea : 4000, Sb = Eb >= 64 ? Eb : 4000;
  bool ok = true;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    if (c == 1) {
      ok = mma::mbar_wait(mma::smem_u32(&sm.done), phase & 1);
      phase += ok ? 1u : 0u;
    }
    const int g = 2 * (tid >> 7);
    store_group(sm.a[0], kRows * 64, mma::swz(a_row(), g), va + 16 * c, Sa);
    store_group(sm.a[0], kRows * 64, mma::swz(a_row(), g + 1), va + 16 * c + 8, Sa);
    if ((warp >> 2) == c) store_group(sm.b[0], kCols * 64, mma::swz(b_col(), warp & 3), vb, Sb);
    mma::fence_async_smem();
    mma::fence_before();
    if (!__syncthreads_and(ok)) return false;
    if (tid == 0) {
      mma::fence_after();
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const uint64_t db = mma::make_desc(mma::smem_u32(sm.b[0]) + 32u * k);
#pragma unroll
        for (int i = 0; i < kDigits; ++i)
          mma::mma_f16(tmem + (uint32_t)(kCols * i), mma::make_desc(mma::smem_u32(sm.a[i]) + 32u * k), db,
                       idesc(kCols * (kDigits - i)), (c > 0 || k > 0 || i > 0) ? 1u : 0u);
      }
      mma::mma_commit(mma::smem_u32(&sm.done));
    }
  }
  ok = mma::mbar_wait(mma::smem_u32(&sm.done), phase & 1);
  phase += ok ? 1u : 0u;
  if (!__syncthreads_and(ok)) return false;
  mma::fence_after();
  // fold: order sums -> T -> FP64
  const int row = 32 * (warp & 3) + lane, c0 = 16 * (warp >> 2);
  const uint32_t base = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0;
  const int er = sm.ea[row];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float o[kDigits][4];
#pragma unroll
    for (int k = 0; k < kDigits; ++k) mma::tmem_ld4(base + (uint32_t)(kCols * k + 4 * q), o[k]);
    mma::tmem_wait_ld();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int ec = sm.eb[c0 + 4 * q + j];
      // orders 0..4 are integers of at most 2^22: their low bits by the magic number 1.5 x 2^23
      int s[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) s[k] = __float_as_int(__fadd_rn(o[k][j], 12582912.0f)) - 0x4B400000;
      const int s5 = __float2int_rn(fmaf(o[6][j], 0.00390625f, fmaf(o[7][j], 1.52587890625e-5f, o[5][j])));
      const int64_t t = (int64_t)(s[2] * 256 + s[3]) * 65536 + (s[4] * 256 + s5) + ((int64_t)(s[0] * 256 + s[1]) << 32);
      const int f = er + ec - 2044 - 52 + 1023;  // exponent field of T's unit
      double& r = acc[4 * q + j];
      if (er >= kBigField || ec >= kBigField)
        r += chain(row, c0 + 4 * q + j);
      else
        r = fma(__ll2double_rn(t), __hiloint2double(f > 0 ? f << 20 : 0, 0), r);
    }
  }
  mma::fence_before();  // the next window's MMAs come after the caller's next barrier
  return true;
}

}  // namespace fx
}  // namespace psq
