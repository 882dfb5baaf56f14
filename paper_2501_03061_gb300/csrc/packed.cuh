// Packed FP32 arithmetic on complex numbers.
#pragma once

#include "common.cuh"

namespace pt {
namespace rl {

// Packed FP32 arithmetic: one instruction for both components of a complex number (each rounded as by
// the scalar instruction).
__device__ __forceinline__ c64 padd(c64 a, c64 b) {
  c64 r;
  asm("{.reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; add.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z;}"
      : "=f"(r.re), "=f"(r.im)
      : "f"(a.re), "f"(a.im), "f"(b.re), "f"(b.im));
  return r;
}
__device__ __forceinline__ c64 pfma(c64 a, float s, c64 c) {  // a * s + c
  c64 r;
  asm("{.reg .b64 x, y, z, w; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %4}; mov.b64 z, {%5, %6}; fma.rn.f32x2 w, x, y, z; mov.b64 {%0, %1}, w;}"
      : "=f"(r.re), "=f"(r.im)
      : "f"(a.re), "f"(a.im), "f"(s), "f"(c.re), "f"(c.im));
  return r;
}
__device__ __forceinline__ c64 psub(c64 a, c64 b) { return pfma(b, -1.f, a); }
__device__ __forceinline__ c64 pmul(c64 a, float s) {
  c64 r;
  asm("{.reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %4}; mul.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z;}"
      : "=f"(r.re), "=f"(r.im)
      : "f"(a.re), "f"(a.im), "f"(s));
  return r;
}
// the same operations in FP64, one component at a time
__device__ __forceinline__ c128 padd(c128 a, c128 b) { return a + b; }
__device__ __forceinline__ c128 psub(c128 a, c128 b) { return a - b; }
__device__ __forceinline__ c128 pfma(c128 a, double s, c128 c) { return {fma(a.re, s, c.re), fma(a.im, s, c.im)}; }
__device__ __forceinline__ c128 pmul(c128 a, double s) { return a * s; }
}  // namespace rl
}  // namespace pt
