// FP64 sums of products on the tensor cores, without rounding the products: per window of 64
// points, R[r][c] += sum_p a_r(p) b_c(p) for a tile of 128 rows x 32 columns, by a CTA of 256
// threads.
//
// GB300's FP64 pipe does two FMAs per clock and SM (1.25 TFLOP/s), its tensor cores 4096 16-bit
// ones.  So every value is cut, without rounding error, into integer digits (the error-free split
// of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59 (2012), here with one power-of-two scale
// per row and window).  With |v| < 2^e over the window, X = trunc(v 2^(63-e)) is a 64-bit integer
// (exact for values above 2^-10 of the window's largest), written as eight balanced base-256
// digits d_k in [-128, 127], exact in FP16.  The products of orders i + j = 0..7 (36 of 64)
// accumulate per order in FP32: an order's sum over 64 points stays within 64 x 8 x 2^14 = 2^23,
// so the accumulation is exact.  The order sums join in one 64-bit integer T and the FP64
// accumulator of an element takes T by one FMA per window: where a chain of FP64 FMAs rounds 64
// times, this rounds once.
//
// What is dropped, of a product of scales S = 2^(e_a + e_b): the seven products of order 8 and those
// above, at most 64 x 7 x 2^14 x 2^-78 (1 + 2^-8) = 2^-55.2 S, and the truncation of small values, at
// most 64 x 2 x 2^-63 = 2^-56 S; typically 2^-61 S.  That is an error relative to the largest values
// of the window, not to an element's own terms.  So a row's bits in `near` mark the points where it is
// above 2^-4 of its scale (kNear), and an element whose two rows share such a point has terms of at
// least 2^-8 S: its error stays within 2^-46.5 of the sum of its absolute terms, about the bound of the
// chain it stands for (63 roundings, 2^-47).  Where the rows share none (two steep functions that
// peak at opposite ends of the window) and the running sum is below S as well (above it, what is
// dropped stays below half a rounding of that sum), the element's window is summed by that chain
// instead: none to one element in 10^5 on grids with whole cells per window, one in 10^3 to 10^2 on
// coarse grids with cells of 27 or 45 points, a quarter of the elements in the RI of a molecule's integrals
// (whose rows are graded).
// Measured (no near bits, no chain -> now): bent triatomic 4.95 -> 5.15 ms, RI of 693 aux functions
// (random) 8.73 -> 8.61 ms, H2 unchanged, 2-centre Coulomb of 18 functions on 7.6 M points (tiles of few rows, bound by
// each window's latency) 11.6 -> 13.6 ms; quintuple-zeta N-O on 8 x 6 x 3 cells of 5 x 3 x 3 points, (P|Q) and
// (P|ij) 4.7 -> 8.6 ms (FP64 FMAs throughout: 28.0).  RI of CO's own integrals (178 aux functions, 3,600 pairs): block
// 0.49 -> 2.3 ms, solve 0.31 -> 0.69 ms (FP64 FMAs: 4.2 and 0.51 ms).
//
// Rows with an infinity, a NaN or a value of 2^478 and above take the chain too (their products may
// leave the range of the integer path).  Rows below 2^-959 (a steep function far out) are lifted by
// 2^200 first, and sums whose unit lies below 2^-1022 are scaled in two steps: nothing is flushed that
// FP64 would keep.
//
// Layout.  Two CTAs per SM (84 KB of shared memory and 256 of the 512 TMEM columns each), so that
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
constexpr int kTogether = 16;           // chains of four columns that the warp sums one by one, all lanes on each
constexpr uint32_t kTmemCols = kDigits * kCols;
constexpr int kBigField = 1500;         // exponent field from which a row takes the FP64 chain
constexpr int kLift = 200;              // power of two by which a row of tiny values is lifted
constexpr int kBias = 256;              // keeps the stored field of a lifted row positive
constexpr int kFar = 8000;              // stored field of a row that always takes the chain
constexpr int kNear = 2;                // a value of a field at most this below its row's counts as large

struct Smem {
  alignas(1024) uint8_t a[kDigits][kRows * 64];
  alignas(1024) uint8_t b[kDigits][kCols * 64];
  int ea[2][kRows], eb[2][kCols];  // exponent fields + kBias, of even and odd windows (0: all zeros)
  alignas(8) uint8_t na[2][kRows][kWin / 8], nb[2][kCols][kWin / 8];  // bit p: the value at point p is large
  alignas(8) uint64_t done;
  uint32_t tmem;
};
constexpr size_t kSmemBytes = sizeof(Smem) + 1024;
static_assert(3 * (kSmemBytes + 1024) > 228 * 1024, "a third CTA per SM would wait for TMEM columns");

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

// The operand values a thread brings to a window.  A: rows a_row(u), u = 0, 1; of chunk c (32
// points) the eight points from a_pt(c): va[2 c + u][i].  B: column b_col(); of chunk c the four
// points from b_pt(c): vb[c][i].  A row's 64 points are in four lanes, a column's in eight.
__device__ __forceinline__ int a_row(int u) { return 64 * u + 8 * (threadIdx.x >> 5) + ((threadIdx.x & 31) >> 2); }
__device__ __forceinline__ int a_pt(int c) { return 32 * c + 8 * (threadIdx.x & 3); }
__device__ __forceinline__ int b_col() { return 4 * (threadIdx.x >> 5) + ((threadIdx.x & 31) >> 3); }
__device__ __forceinline__ int b_pt(int c) { return 32 * c + 4 * (threadIdx.x & 7); }

// Biased digits of v (byte k of the result = digit 7 - k plus 128) in a window whose largest
// exponent field is E (E = 4000: a row of zeros).  near takes a bit at its low end: v is large.
__device__ __forceinline__ uint64_t digits(double v, int E, uint32_t& near) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const int t = min(E - (int)((hi >> 20) & 0x7ffu), 63);
  near = __funnelshift_l((uint32_t)(t - 2 - kNear), near, 1);  // (the difference's sign)
  const uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  const uint64_t x = (m << 10) >> t;
  const uint64_t s = (uint64_t)((int64_t)(int32_t)hi >> 63);
  return (x ^ s) + (0x8080808080808080ull - s);
}

// Digit plane k of the biased digits y0, y1 as two FP16 numbers: 1024 + byte, minus 1152.
__device__ __forceinline__ uint32_t plane(uint64_t y0, uint64_t y1, int k) {
  const uint32_t u0 = k < 4 ? (uint32_t)(y0 >> 32) : (uint32_t)y0, u1 = k < 4 ? (uint32_t)(y1 >> 32) : (uint32_t)y1;
  const uint32_t by = 3 - (k & 3);
  const uint32_t x = (__byte_perm(u0, u1, by | (by << 4) | ((4 + by) << 8) | ((4 + by) << 12)) & 0x00ff00ffu) | 0x64006400u;
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&x), __half2half2(__ushort_as_half(0x6480)));
  return *reinterpret_cast<const uint32_t*>(&d);
}

// Eight consecutive points of a row into its 16-byte group of every plane (offset off); their near bits.
__device__ __forceinline__ uint32_t store_a(Smem& sm, uint32_t off, const double (&v)[8], int E) {
  uint64_t y[8];
  uint32_t near = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) y[i] = digits(v[i], E, near);
#pragma unroll
  for (int k = 0; k < kDigits; ++k)
    *reinterpret_cast<uint4*>(sm.a[k] + off) =
        make_uint4(plane(y[0], y[1], k), plane(y[2], y[3], k), plane(y[4], y[5], k), plane(y[6], y[7], k));
  return near;
}

// Four consecutive points of a column into their half group.
__device__ __forceinline__ uint32_t store_b(Smem& sm, uint32_t off, const double (&v)[4], int E) {
  uint64_t y[4];
  uint32_t near = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) y[i] = digits(v[i], E, near);
#pragma unroll
  for (int k = 0; k < kDigits; ++k)
    *reinterpret_cast<uint2*>(sm.b[k] + off) = make_uint2(plane(y[0], y[1], k), plane(y[2], y[3], k));
  return near;
}

__device__ __forceinline__ int hi_abs(double v) { return __double2hiint(v) & 0x7fffffff; }
// The size of v as an integer: exponent and the mantissa's first 21 bits (0 below 2^-1043: low_bits).
__device__ __forceinline__ uint32_t mag(double v) {
  return __funnelshift_l((uint32_t)__double2loint(v), (uint32_t)__double2hiint(v), 1);
}
__device__ __forceinline__ uint32_t low_bits(double v) { return (uint32_t)__double2loint(v); }
// The exponent field a window is scaled by, from its largest size: one more where the largest value is within
// 2^-7 of the next power of two (its leading digit would round up to 128).  A NaN's payload counts for
// nothing (the sum would wrap).
__device__ __forceinline__ int field(uint32_t mx) { return (int)((min(mx, 0xffe00000u) + 0x4080u) >> 21); }
constexpr uint32_t kLow = 64u << 21;  // rows below it are lifted

// What a row's or column's window is scaled by: the field its digits are cut with (kZeros for zeros: their
// own field, 0, must be 63 below it) and the stored one.
constexpr int kZeros = 4000;
__device__ __forceinline__ int digit_field(uint32_t mx) { return mx == 0 ? kZeros : field(mx); }
__device__ __forceinline__ int stored_field(uint32_t mx, bool lifted) {
  const int E = field(mx);
  return mx == 0 ? 0 : (E >= kBigField ? kFar : E + kBias - (lifted ? kLift : 0));
}
// The near bits as the fold wants them: zeros meet anything, rows out of the digits' range nothing.
__device__ __forceinline__ uint32_t near_bits(uint32_t near, int E) { return E < kBigField ? near : (E == kZeros ? ~0u : 0u); }

// The chains of a warp's 32 rows and 16 columns, added to its sums (bit j of apart: this lane's row with column
// c0 + j), four columns at a time: few of them one by one by all lanes (two points a lane), more by
// their own lanes, four columns' operands in flight.  A function of its own, on a copy of the sums, so that
// what it needs stays out of the window's registers.
template <typename Chain>
__device__ __noinline__ void chains(Chain chain, double* sums, uint32_t apart, int row0, int c0) {
  constexpr unsigned kFull = 0xffffffffu;
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int q = 0; q < 16; q += 4, apart >>= 4) {
    uint32_t m[4];
    int count = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      m[j] = __ballot_sync(kFull, apart >> j & 1);
      count += __popc(m[j]);
    }
    if (count > kTogether) {
      double s[4] = {};
      if (apart & 15u) chain(row0 + lane, c0 + q, 0, 1, s);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (apart >> j & 1) sums[q + j] += s[j];
      __syncwarp();
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll 1
        for (; m[j]; m[j] &= m[j] - 1) {
          const int l = __ffs(m[j]) - 1;
          double s[1] = {};
          chain(row0 + l, c0 + q + j, lane, 32, s);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) s[0] += __shfl_xor_sync(kFull, s[0], o);
          if (l == lane) sums[q + j] += s[0];
        }
    }
  }
}

// One window: the tile's accumulators (element row 32 (warp % 4) + lane, columns 16 (warp / 4) + j,
// acc[j]) take sum_p a_r(p) b_c(p).  Only the first `rows` rows and `cols` columns are kept up
// (8-row groups and 4-column groups past them are left out).  win: the windows done so far by this
// CTA.  chain(row, col, p, step, s): the plain FP64 sums of the window's points p, p + step, ... for a row and the
// s's size of columns from col, for rows or columns out of the integer
// path's range and for an element whose rows are not large at a common point.  ok turns false when a wait ran out (the caller ends its loop when the return
// value, the same for all threads, is false, and asks all threads once more at the end).
template <typename Chain>
__device__ __forceinline__ bool window(Smem& sm, uint32_t tmem, double (&va)[4][8], double (&vb)[2][4],
                                       double (&acc)[16], uint32_t& phase, uint32_t win, int rows, int cols, bool& ok,
                                       Chain chain, uint64_t wait_ns = mma::kWaitNs) {
  constexpr unsigned kFull = 0xffffffffu;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int set = win & 1;
  auto over_a = [&](int u, auto part) {  // the largest part of row u's values
    uint32_t m = 0;
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int i = 0; i < 8; ++i) m = max(m, part(va[2 * c + u][i]));
    m = max(m, __shfl_xor_sync(kFull, m, 1));
    return max(m, __shfl_xor_sync(kFull, m, 2));
  };
  auto over_b = [&](auto part) {
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) m = max(m, max(part(vb[0][i]), part(vb[1][i])));
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) m = max(m, __shfl_xor_sync(kFull, m, o));
    return m;
  };
  uint32_t ma[2] = {over_a(0, mag), over_a(1, mag)}, mb = over_b(mag);
  // small rows: those that are not zero (also below 2^-1043) are lifted
  bool la0 = false, la1 = false, lb = false;
  if (__any_sync(kFull, (ma[0] < kLow && a_row(0) < rows) || (ma[1] < kLow && a_row(1) < rows) || (mb < kLow && b_col() < cols))) {
    const uint32_t wa0 = over_a(0, low_bits), wa1 = over_a(1, low_bits), wb = over_b(low_bits);  // (all lanes shuffle)
    la0 = ma[0] < kLow && (ma[0] | wa0) != 0;
    la1 = ma[1] < kLow && (ma[1] | wa1) != 0;
    lb = mb < kLow && (mb | wb) != 0;
    if (__any_sync(kFull, la0 || la1 || lb)) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          va[2 * c][i] *= la0 ? 0x1p200 : 1.0;
          va[2 * c + 1][i] *= la1 ? 0x1p200 : 1.0;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) vb[c][i] *= lb ? 0x1p200 : 1.0;
      }
      ma[0] = over_a(0, mag);
      ma[1] = over_a(1, mag);
      mb = over_b(mag);
    }
  }
  const int ea[2] = {digit_field(ma[0]), digit_field(ma[1])}, eb = digit_field(mb);
  if ((lane & 3) == 0) {
    sm.ea[set][a_row(0)] = stored_field(ma[0], la0);
    sm.ea[set][a_row(1)] = stored_field(ma[1], la1);
  }
  if ((lane & 7) == 0) sm.eb[set][b_col()] = stored_field(mb, lb);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    if (c == 1 && ok) {
      ok = mma::mbar_wait(mma::smem_u32(&sm.done), phase & 1, nullptr, wait_ns);
      phase += ok ? 1u : 0u;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (64 * u + 8 * warp < rows) {
        const uint32_t near = store_a(sm, mma::swz(a_row(u), lane & 3), va[2 * c + u], ea[u]);
        sm.na[set][a_row(u)][4 * c + (lane & 3)] = (uint8_t)near_bits(near, ea[u]);
      }
    if (4 * warp < cols) {
      uint32_t near = near_bits(store_b(sm, mma::swz(b_col(), (lane & 7) >> 1) + 8u * (lane & 1), vb[c], eb), eb) & 15u;
      near = (near << 4) | __shfl_down_sync(kFull, near, 1);  // the pair's first points in the high bits, as in na
      if ((lane & 1) == 0) sm.nb[set][b_col()][4 * c + ((lane & 7) >> 1)] = (uint8_t)near;
    }
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
  ok = mma::mbar_wait(mma::smem_u32(&sm.done), phase & 1, nullptr, wait_ns);
  phase += ok ? 1u : 0u;
  if (!__all_sync(kFull, ok)) { ok = false; return true; }
  mma::fence_after();
  // fold: order sums -> T -> FP64
  const int row = 32 * (warp & 3) + lane, c0 = 16 * (warp >> 2);
  if (32 * (warp & 3) < rows) {
    const uint32_t base = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0;
    const int er = sm.ea[set][row];
    const uint2 near = row < rows ? *reinterpret_cast<const uint2*>(sm.na[set][row]) : make_uint2(~0u, ~0u);
    uint32_t apart = 0;  // bit j: element j takes the chain
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (c0 + 4 * q >= cols) break;
      float o[kDigits][4];
      __syncwarp();
#pragma unroll
      for (int k = 0; k < kDigits; ++k) mma::tmem_ld4(base + (uint32_t)(kCols * k + 4 * q), o[k]);
      mma::tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int ec = sm.eb[set][c0 + 4 * q + j];
        const uint2 nc = *reinterpret_cast<const uint2*>(sm.nb[set][c0 + 4 * q + j]);
        // orders 0..3 are integers of at most 2^22: their low bits by the magic number 1.5 x 2^23
        int s[6];
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] = __float_as_int(__fadd_rn(o[k][j], 12582912.0f)) - 0x4B400000;
        s[4] = __float2int_rn(o[4][j]);
        s[5] = __float2int_rn(o[5][j]);
        // orders 0..5 in units of order 5 (at most 2^61); orders 6 and 7 join in those units where
        // the sum is large, in 1/128 of them where it is below 2^54 (a sum of cancelling terms)
        int64_t t = (int64_t)(s[2] * 256 + s[3]) * 65536 + (s[4] * 256 + s[5]) + ((int64_t)(s[0] * 256 + s[1]) << 32);
        const bool small = (uint32_t)((int)(t >> 32) + (1 << 22)) < (1u << 23);
        t = (small ? t << 7 : t) +
            __float2int_rn(fmaf(o[6][j], 0.00390625f, o[7][j] * 1.52587890625e-5f) * (small ? 128.0f : 1.0f));
        int f = er + ec - 2 * kBias - 2044 - 54 + 1023 - (small ? 7 : 0);  // exponent field of t's unit
        // t as FP64; where its unit lies below 2^-1022, 2^600 go over from t (by its exponent bits: the FP64
        // pipe is the scarce one) to the unit
        const double x = __ll2double_rn(t);
        int hx = __double2hiint(x);
        if (f <= 0) {
          hx -= t == 0 ? 0 : 600 << 20;
          f = max(f + 600, 0);
        }
        // no common large point, and the running sum below S
        if (((near.x & nc.x) | (near.y & nc.y)) == 0 &&
            (hi_abs(acc[4 * q + j]) >> 20) < er + ec - 2 * kBias - 2044 + 1023)
          apart |= 1u << (4 * q + j);
        else
          acc[4 * q + j] = fma(__hiloint2double(hx, __double2loint(x)), __hiloint2double(f << 20, 0), acc[4 * q + j]);
      }
    }
    if (__any_sync(kFull, apart)) {
      double sums[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) sums[j] = acc[j];
      chains(chain, sums, apart, row - lane, c0);
#pragma unroll
      for (int j = 0; j < 16; ++j) acc[j] = sums[j];
    }
  }
  mma::fence_before();  // the next window's MMAs come after its first barrier
  return true;
}

}  // namespace fx
}  // namespace psq
