// Two float32 values in one 64-bit register pair, with the packed directed
// arithmetic of sm_103a (fma / add / mul .rp.f32x2): one instruction for two
// independent operations.  The pipe's rate in operations is the same
// (measured: 74 TFLOP/s scalar, 70 packed), but it takes half the issue slots,
// which is what bounds the kernels here: in-register line transforms of
// order 8 need 52% of the instructions.
//
// The kernels hold a pair of bounds as (negated lower, upper): with
// RD(x) = -RU(-x), rounding up serves both and every value is bit for bit the
// one a round-down instruction gives.
#pragma once

#include <cuda_runtime.h>

namespace bern {

typedef unsigned long long p2;

__device__ __forceinline__ p2 pack2(float a, float b) {
  p2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(p2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ p2 fma2_ru(p2 a, p2 b, p2 c) {
  p2 r;
  asm("fma.rp.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ p2 add2_ru(p2 a, p2 b) {
  p2 r;
  asm("add.rp.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ p2 mul2_ru(p2 a, p2 b) {
  p2 r;
  asm("mul.rp.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

}  // namespace bern
