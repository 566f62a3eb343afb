// Float pairs in one 64-bit register for the float32 passes: the packed add,
// multiply and multiply-add of this GPU (one instruction for two float32
// operations, each rounded as its scalar form).  Packing saves issue slots, not
// float32 throughput; the passes over the neighbour list are bound by issue.
#pragma once

#include <cuda_runtime.h>

#include "device_common.cuh"

namespace apip {

struct F2 { unsigned long long v; };
__device__ __forceinline__ F2 f2(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ F2 f2(float a) { return f2(a, a); }
__device__ __forceinline__ float2 f2_get(F2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
// a - b, exactly rounded (the product b * -1 is exact)
__device__ __forceinline__ F2 sub2(F2 a, F2 b) { return fma2(b, f2(-1.f), a); }
__device__ __forceinline__ F2 clamp2(F2 a) {   // to [-1, 1]
  const float2 v = f2_get(a);
  return f2(fminf(1.f, fmaxf(-1.f, v.x)), fminf(1.f, fmaxf(-1.f, v.y)));
}
// exp(x) as 2^(x log2 e) on the hardware's base-2 exponential
__device__ __forceinline__ F2 exp2x(F2 x) {
  const float2 v = f2_get(mul2(x, f2(1.44269504f)));
  float a, b;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(v.x));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(v.y));
  return f2(a, b);
}
__device__ __forceinline__ F2 rsqrt2(F2 x) {
  const float2 v = f2_get(x);
  float a, b;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(v.x));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(v.y));
  return f2(a, b);
}

// The quintic taper f_trans at r (Eq. S1, in the factored form of ftrans), without
// its two early returns: t clamped to [-1, 1] gives 1 and 0 exactly, and a zero
// derivative, at the ends (and 0 for a NaN).  c = lo + hi, iw = 1 / (hi - lo).
__device__ __forceinline__ F2 taper_t(F2 r, F2 c, F2 iw) { return clamp2(mul2(fma2(f2(-2.f), r, c), iw)); }
__device__ __forceinline__ F2 taper_f(F2 t) {
  const F2 p = add2(f2(1.f), t);
  return mul2(mul2(mul2(mul2(f2(0.0625f), p), p), p), fma2(t, fma2(f2(3.f), t, f2(-9.f)), f2(8.f)));
}
// derivative with respect to r; dw = -2 iw
__device__ __forceinline__ F2 taper_df(F2 t, F2 dw) {
  const F2 u = fma2(t, t, f2(-1.f));   // -(1 - t^2); its sign cancels in the square
  return mul2(mul2(mul2(f2(0.9375f), u), u), dw);
}

// Two running sums with Kahan's compensation (Acc), the compensation kept with its
// sign turned (n = -c) so that a product enters with one multiply-add.
struct Acc2 {
  F2 s, n;
  __device__ __forceinline__ Acc2() : s(f2(0.f)), n(f2(0.f)) {}
  __device__ __forceinline__ void add_y(F2 y) {   // y = value + n
    const F2 t = add2(s, y);
    n = sub2(y, sub2(t, s));
    s = t;
  }
  __device__ __forceinline__ void add(F2 v) { add_y(add2(v, n)); }
  __device__ __forceinline__ void add_prod(F2 a, F2 b) { add_y(fma2(a, b, n)); }
  // both sums and what they still have to give back, over the LANES threads of an atom
  template <int LANES>
  __device__ __forceinline__ float value() const {
    const float2 a = f2_get(s), b = f2_get(n);
    FF f = ff_sum(a.x, a.y);
    f.lo += b.x + b.y;
#pragma unroll
    for (int o = 1; o < LANES; o <<= 1)
      f = ff_add(f, FF{__shfl_xor_sync(0xffffffffu, f.hi, o), __shfl_xor_sync(0xffffffffu, f.lo, o)});
    return f.hi + f.lo;
  }
};
// a plain pair of sums, added up over the LANES threads of an atom
template <int LANES>
__device__ __forceinline__ float sum2(F2 a) {
  const float2 v = f2_get(a);
  float s = v.x + v.y;
#pragma unroll
  for (int o = 1; o < LANES; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

}  // namespace apip
