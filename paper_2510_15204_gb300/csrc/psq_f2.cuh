// Packed FP32 arithmetic: two IEEE single-precision operations per instruction (sm_100 and up), each
// half rounded to nearest as the scalar instruction does.  A packed instruction takes one issue slot
// and one instruction fetch for two results; the kernels that use it are bound by those.
#pragma once
#include <cstdint>

namespace psq {

struct f2 {
  uint64_t v;
};

__device__ __forceinline__ f2 f2_pack(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f2 f2_both(float x) { return f2_pack(x, x); }
__device__ __forceinline__ void f2_unpack(f2 a, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
// b - a (the product by -1 is exact)
__device__ __forceinline__ f2 f2_rsub(f2 a, f2 b) { return f2_fma(a, f2_both(-1.0f), b); }

}  // namespace psq
