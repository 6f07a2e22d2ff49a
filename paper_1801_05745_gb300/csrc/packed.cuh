// Packed FP32 arithmetic (two values per 64-bit register), shared by the
// double-float kernels.
#pragma once
#include <cuda_runtime.h>

namespace ufc {

// Two double-floats side by side in the packed FP32 instructions of sm_100
// and later (add/sub/mul/fma.rn.f32x2: one issue slot for two correctly
// rounded FP32 operations).  Kernels bound by the FP32 pipe are, with scalar
// instructions, bound by the issue slots as well; packing two values leaves
// slots for the loads, shuffles and votes around the arithmetic.  Measured on
// chains of independent operations: fma 37.1 T lane operations/s packed and
// 36.6 scalar, add and mul 37.1 packed and 35.1 scalar at 32 warps per SM; at 8
// warps per SM 34.4 packed against 28 scalar.
typedef unsigned long long u64;
__device__ __forceinline__ u64 x2_pack(float a, float b) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 x2_get(u64 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ u64 x2_add(u64 a, u64 b) {
  u64 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 x2_sub(u64 a, u64 b) {
  u64 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 x2_mul(u64 a, u64 b) {
  u64 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 x2_fma(u64 a, u64 b, u64 c) {
  u64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ u64 x2_neg(u64 a) { return a ^ 0x8000000080000000ull; }
struct dfx { u64 h, l; };

// a + b, the low part not renormalised
__device__ __forceinline__ dfx dfx_add_raw(dfx a, dfx b) {
  const u64 s = x2_add(a.h, b.h);
  const u64 bb = x2_sub(s, a.h);
  const u64 er = x2_add(x2_sub(a.h, x2_sub(s, bb)), x2_sub(b.h, bb));
  return {s, x2_add(er, x2_add(a.l, b.l))};
}
// h + l renormalised (|h| >= |l|)
__device__ __forceinline__ dfx dfx_norm(u64 h, u64 l) {
  const u64 s = x2_add(h, l);
  return {s, x2_sub(l, x2_sub(s, h))};
}
// a * b, renormalised.  (With the product of the low parts: left out, a square is
// too small by 2^-49 of itself on average.)
__device__ __forceinline__ dfx dfx_mul(dfx a, dfx b) {
  const u64 p = x2_mul(a.h, b.h);
  u64 e = x2_fma(a.h, b.h, x2_neg(p));
  e = x2_fma(a.h, b.l, e);
  e = x2_fma(a.l, b.h, e);
  return dfx_norm(p, x2_fma(a.l, b.l, e));
}

}  // namespace ufc
