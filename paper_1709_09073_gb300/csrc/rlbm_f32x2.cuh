// Packed pairs of FP32 values (the f32x2 instructions of sm_100 and later): one issue
// slot for two FP32 operations. The pair occupies the FP32 pipe for two clocks
// (measured 2.15 with a constant or broadcast operand, 3.2 with three register
// pairs, against 1.2 and 1.75 for one scalar FMA), so it saves issue slots, not pipe
// time: it pays where a kernel is bound by its instruction count. A broadcast
// (f2_dup of a register or a constant) and a negation are free, folded into the operand.
#pragma once
#include <cuda_runtime.h>

namespace rlbm {

struct f2 {
  unsigned long long v;
};

__device__ __forceinline__ f2 f2_make(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ f2 f2_dup(float a) { return f2_make(a, a); }
__device__ __forceinline__ void f2_split(f2 a, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
}
__device__ __forceinline__ float f2_lo(f2 a) {
  float x, y;
  f2_split(a, x, y);
  return x;
}
__device__ __forceinline__ float f2_hi(f2 a) {
  float x, y;
  f2_split(a, x, y);
  return y;
}

// The same names on scalars and pairs, each operation rounded to nearest and never
// contracted with a neighbour.
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ f2 vfma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ f2 vmul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 vadd(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 vsub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 vneg(f2 a) {
  float x, y;
  f2_split(a, x, y);
  return f2_make(-x, -y);
}

}  // namespace rlbm
