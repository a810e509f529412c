// Packed FP32 pairs: two FP32 values in one 64-bit register and the packed
// add / mul / fma of sm_100 and later (PTX .f32x2).  One instruction gives two
// results at the scalar operation's rate per result (measured on GB300,
// microbench/alu_peaks.cu: an fma whose three register operands are its own takes
// 1.5 cycles of a scheduler, the packed one three for its two results, an add or
// mul one a result), so a kernel bound by instruction
// issue rather than by the FMA pipe runs two independent evaluations in the
// issue slots of one.  Rounding is that of the scalar operation (.rn), and
// an fma is a fused multiply-add exactly as fmaf.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace bipb {

struct f2 {
  unsigned long long v;
};

__device__ __forceinline__ f2 f2_make(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f2 f2_splat(float a) { return f2_make(a, a); }
__device__ __forceinline__ void f2_get(f2 a, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
// the two values added
__device__ __forceinline__ float f2_sum(f2 a) {
  float lo, hi;
  f2_get(a, lo, hi);
  return lo + hi;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
// a * b + c
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

}  // namespace bipb
