// The codelets' arithmetic (fft_reg.cuh) on packed single-precision pairs.
#pragma once

#include "fft_reg.cuh"

namespace kss {
namespace fftr {

// Single precision with both components in one packed instruction where the operation does not mix them
// (the passes that use it are bound by issue slots; middle pass of 564 bands at 96 points 1.78 -> 1.70
// ms).  Swapped components stay with the scalar operations, where the swap is free.  A type of its own:
// it rounds differently in the last bit where the compiler contracts the scalar form across additions,
// and the single-precision density, delivered in FP64, keeps the scalar form.
struct alignas(8) F2 {
  float x, y;
  F2() = default;
  __device__ __forceinline__ F2(float a, float b) : x(a), y(b) {}
  __device__ __forceinline__ F2(float2 a) : x(a.x), y(a.y) {}
  __device__ __forceinline__ operator float2() const { return make_float2(x, y); }
};
template <typename C> struct Packed { using T = C; };
template <> struct Packed<float2> { using T = F2; };
__device__ __forceinline__ F2 add(F2 a, F2 b) {
  F2 r;
  asm("{.reg .b64 p, q, s; mov.b64 p, {%2, %3}; mov.b64 q, {%4, %5}; add.rn.f32x2 s, p, q; mov.b64 {%0, %1}, s;}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ F2 sub(F2 a, F2 b) {
  F2 r;
  asm("{.reg .b64 p, q, s; mov.b64 p, {%2, %3}; mov.b64 q, {%4, %5}; sub.rn.f32x2 s, p, q; mov.b64 {%0, %1}, s;}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ F2 axpy(float a, F2 b, F2 c) {
  F2 r;
  asm("{.reg .b64 p, q, s, t; mov.b64 p, {%2, %2}; mov.b64 q, {%3, %4}; mov.b64 s, {%5, %6};"
      " fma.rn.f32x2 t, p, q, s; mov.b64 {%0, %1}, t;}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}
__device__ __forceinline__ F2 scaled(float a, F2 b) {
  F2 r;
  asm("{.reg .b64 p, q, s; mov.b64 p, {%2, %2}; mov.b64 q, {%3, %4}; mul.rn.f32x2 s, p, q; mov.b64 {%0, %1}, s;}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ F2 add_i(F2 a, F2 d, float s) {
  return s > 0.f ? F2(a.x - d.y, a.y + d.x) : F2(a.x + d.y, a.y - d.x);
}
__device__ __forceinline__ F2 sub_i(F2 a, F2 d, float s) { return add_i(a, d, -s); }
__device__ __forceinline__ F2 mul(F2 a, float2 b) { return mul(a, F2(b)); }

}  // namespace fftr
}  // namespace kss
