// f32x2.cuh -- packed FP32 pairs (add/sub/mul/fma .f32x2: one instruction
// for two lanes of data on GB300) and a TwoSum accumulator on pairs.
#pragma once

namespace whff {
namespace dev {

// Packed FP32 pairs (add/sub/mul/fma .f32x2, one instruction for two lanes
// of data): each half rounds exactly like the scalar instruction.  The
// compiler may fuse a packed multiply into a packed add that consumes it, so
// a product whose rounding matters is formed with scalar __fmul_rn instead.
__device__ __forceinline__ float2 add_f2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "add.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}\n"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 sub_f2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "sub.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}\n"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 mul_f2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "mul.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}\n"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 fma_f2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, c, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "mov.b64 c, {%6, %7};\n\tfma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}\n"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}

// two_sum_acc on a pair of accumulators
__device__ __forceinline__ void two_sum_acc2(float2& hi, float2& lo, float2 p) {
  const float2 s = add_f2(hi, p);
  const float2 bp = sub_f2(s, hi);
  const float2 err = add_f2(sub_f2(hi, sub_f2(s, bp)), sub_f2(p, bp));
  hi = s;
  lo = add_f2(lo, err);
}

// The same pairs held as 64-bit registers across a loop.
using f32p = unsigned long long;
__device__ __forceinline__ f32p pair_of(float a, float b) {
  f32p d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float2 halves_of(f32p a) {
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(a));
  return d;
}
__device__ __forceinline__ f32p add_p(f32p a, f32p b) {
  f32p d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32p sub_p(f32p a, f32p b) {
  f32p d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32p fma_p(f32p a, f32p b, f32p c) {
  f32p d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
// TwoSum of q s into (hi, lo), s a power of two: the product is exact, so the
// scaling rides in two of the FMAs (-bp = hi - s' is as exact as bp).
__device__ __forceinline__ void two_sum_scaled_p(f32p& hi, f32p& lo, f32p q, f32p s) {
  const f32p t = fma_p(q, s, hi), nbp = sub_p(hi, t);
  const f32p err = add_p(sub_p(hi, add_p(t, nbp)), fma_p(q, s, nbp));
  hi = t;
  lo = add_p(lo, err);
}

}  // namespace dev
}  // namespace whff
