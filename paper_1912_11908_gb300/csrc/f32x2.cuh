// Pairs of FP32 values in one 64-bit register: Blackwell's packed FP32 add, multiply and fused multiply-add work on
// both halves in one instruction, each half rounded as the scalar operation.  They take the arithmetic of kernels that
// are bound by issue slots at half the slots; everything else (reciprocal, square root, minimum, select) takes the
// halves one by one, which costs no moves.
#pragma once

namespace ibm {

struct f2 {
  float x, y;
};

__device__ __forceinline__ float2 raw2(f2 a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ f2 wrap2(float2 a) { return f2{a.x, a.y}; }
__device__ __forceinline__ f2 both(float a) { return f2{a, a}; }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return wrap2(__ffma2_rn(raw2(a), raw2(b), raw2(c))); }
__device__ __forceinline__ f2 fma2(float a, f2 b, f2 c) { return fma2(both(a), b, c); }
__device__ __forceinline__ f2 operator+(f2 a, f2 b) { return wrap2(__fadd2_rn(raw2(a), raw2(b))); }
__device__ __forceinline__ f2 operator+(float a, f2 b) { return both(a) + b; }
__device__ __forceinline__ f2 operator*(f2 a, f2 b) { return wrap2(__fmul2_rn(raw2(a), raw2(b))); }
__device__ __forceinline__ f2 operator*(float a, f2 b) { return both(a) * b; }
__device__ __forceinline__ f2 operator-(f2 a, f2 b) {
  unsigned long long r;
  asm("{ .reg .b64 a, b; mov.b64 a, {%1, %2}; mov.b64 b, {%3, %4}; sub.rn.ftz.f32x2 %0, a, b; }"
      : "=l"(r)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  f2 o;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));
  return o;
}
__device__ __forceinline__ f2 rcp2(f2 a) { return f2{__fdividef(1.f, a.x), __fdividef(1.f, a.y)}; }
__device__ __forceinline__ f2 sqrt2(f2 a) { return f2{sqrtf(a.x), sqrtf(a.y)}; }
__device__ __forceinline__ f2 max2(f2 a, f2 b) { return f2{fmaxf(a.x, b.x), fmaxf(a.y, b.y)}; }
__device__ __forceinline__ f2 min2(f2 a, f2 b) { return f2{fminf(a.x, b.x), fminf(a.y, b.y)}; }
__device__ __forceinline__ f2 ld2(const float *p) {  // 8-byte aligned
  const float2 v = *reinterpret_cast<const float2 *>(p);
  return f2{v.x, v.y};
}
__device__ __forceinline__ void st2(float *p, f2 a) { *reinterpret_cast<float2 *>(p) = make_float2(a.x, a.y); }

}  // namespace ibm
