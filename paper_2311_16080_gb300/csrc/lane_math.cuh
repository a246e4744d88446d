// FP32 arithmetic with every rounding spelled out, for one cell (float) or
// two cells at once (F2, the packed FP32 instructions of sm_100 and later:
// one issue slot for both lanes, each lane rounded like its scalar form).
//
// The collision is written with these, not with operators: which products the
// compiler would fuse into an FMA then depends on the code around them, and a
// cell's result on the kernel (and on how many cells a thread takes) that
// computed it.  Spelled out, every kernel gives the same bits.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace xlb {

struct F2 {
  unsigned long long v;
};

__device__ __forceinline__ F2 pack2(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(F2 a, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
}

template <typename T>
__device__ __forceinline__ T vset(float x);
template <>
__device__ __forceinline__ float vset<float>(float x) {
  return x;
}
template <>
__device__ __forceinline__ F2 vset<F2>(float x) {
  return pack2(x, x);
}

__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vneg(float a) { return -a; }  // (a modifier of the operand that uses it)
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float vrcp(float a) { return 1.0f / a; }

__device__ __forceinline__ F2 vadd(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 vmul(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
// a - b = fma(b, -1, a): one rounding, like the subtraction
__device__ __forceinline__ F2 vsub(F2 a, F2 b) { return vfma(b, pack2(-1.0f, -1.0f), a); }
__device__ __forceinline__ F2 vneg(F2 a) { return vmul(a, pack2(-1.0f, -1.0f)); }
__device__ __forceinline__ F2 vrcp(F2 a) {
  float x, y;
  unpack2(a, x, y);
  return pack2(1.0f / x, 1.0f / y);
}

// a / b by the fast division (CUDA's __fdividef)
__device__ __forceinline__ float vdiv_fast(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ F2 vdiv_fast(F2 a, F2 b) {
  float x, y, z, w;
  unpack2(a, x, y);
  unpack2(b, z, w);
  return pack2(__fdividef(x, z), __fdividef(y, w));
}
// b < lim ? x : c - a / b per lane; no division where none is used
__device__ __forceinline__ float vsub_div_unless_less(float x, float c, float a, float b, float lim) {
  return b < lim ? x : __fsub_rn(c, __fdiv_rn(a, b));
}
__device__ __forceinline__ F2 vsub_div_unless_less(F2 x, float c, F2 a, F2 b, F2 lim) {
  float x0, x1, a0, a1, b0, b1, l0, l1;
  unpack2(x, x0, x1);
  unpack2(a, a0, a1);
  unpack2(b, b0, b1);
  unpack2(lim, l0, l1);
  return pack2(vsub_div_unless_less(x0, c, a0, b0, l0), vsub_div_unless_less(x1, c, a1, b1, l1));
}

}  // namespace xlb
